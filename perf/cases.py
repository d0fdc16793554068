"""Performance cases of the framework: what its users have it do, through its public entry points.

Three kinds of work, each with the sizes of the configurations, tests and benchmark of this repository:

  expert   denoising steps of a whole action expert (`ActionExpert.step`): chunk <- noise, then `steps` Euler steps, optionally
           behind the ring append of a control tick; called directly or replayed from the CUDA graph that a control loop keeps
  path     the layer calls by themselves for callers with projections of their own: ring append, the gates of all layers,
           AdaRMSNorm and partitioned attention per layer, Euler update
  prefix   a new observation: the static prefix of some streams rewritten in place, or staged into the idle bank and committed

Everything a case holds is a plain value; `prepare` draws all inputs from the seed on the GPU.
"""
from __future__ import annotations

import torch

from paper_2607_14695_b200 import binding as rb
from paper_2607_14695_b200 import synth
from paper_2607_14695_b200.expert import ActionExpert, random_weights_device

DEV = "cuda:0"

# one pi0-class action expert (8 query heads on one KV head of 256, chunk of 50, 816-token prefix, ring of 32)
EXPERT = dict(kind="expert", dtype="bf16", B=1, L=18, Hq=8, Hkv=1, d=256, S=816, ragged=False, N=32, T=50, D=1024, F=4096, Cd=288, Hd=256,
              A=32, steps=1, m=0, graph=False)
PATH = dict(kind="path", dtype="bf16", B=1, L=2, Hq=8, Hkv=1, d=256, S=816, ragged=False, N=32, T=50, D=1024, Cd=288, Hd=256, A=32, steps=1, m=0,
            causal=False, outliers=False)
PREFIX = dict(kind="prefix", dtype="bf16", B=8, n=8, L=18, Hkv=1, d=256, S=816, N=32, staged=False)


def listed():
    return [
        # the smallest control tick: one small fp32 layer, one token appended, 4 Euler steps (latency and launches)
        dict(PATH, name="tick_tiny_fp32", dtype="f32", L=1, Hq=2, d=64, S=64, N=16, T=8, D=128, Cd=40, Hd=32, A=8, steps=4, m=1),
        # one robot: the 50 Hz control tick as a control loop runs it, append + 10 steps in one graph replay
        dict(EXPERT, name="tick_1_stream", steps=10, m=1, graph=True),
        # one robot: a denoising step called directly (first tick, changing buffers, no graph)
        dict(EXPERT, name="step_1_direct"),
        # a few robots on one server, graph replay
        dict(EXPERT, name="step_4_streams", B=4, graph=True),
        # an uneven batch: odd number of streams, odd chunk, prefixes of different lengths, called directly
        dict(EXPERT, name="step_13_ragged", B=13, T=33, S=777, ragged=True),
        # batched serving
        dict(EXPERT, name="step_64_streams", B=64, graph=True),
        # batched serving for a caller with its own projections: AdaRMSNorm + partitioned attention per layer
        dict(PATH, name="path_64_streams", B=64, L=4),
        # long context with outliers in the norm input
        dict(PATH, name="path_long_context", B=16, S=4160, N=256, outliers=True),
        # sliding window of ten frames, one frame of 256 tokens appended, long chunk
        dict(PATH, name="path_frames_16", B=16, N=2560, T=100, m=256),
        # one stream over fifty frames
        dict(PATH, name="path_frames_1", B=1, N=12800, T=50, m=256),
        # smaller heads, several KV heads, causal suffix
        dict(PATH, name="path_heads_128", B=6, L=4, Hq=16, Hkv=4, d=128, S=300, ragged=True, N=48, T=37, D=2048, m=3, causal=True),
        # a new observation for eight streams, staged beside the running steps and committed
        dict(PREFIX, name="prefix_staged_8", staged=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["expert", "expert", "expert", "path", "path", "path", "path", "prefix"])
    if kind == "expert":
        B = _log_int(rng, 1, 64)
        c = dict(EXPERT, B=B, T=rng.randint(20, 50) if rng.random() < 0.5 else 50, S=rng.randint(300, 816), ragged=rng.random() < 0.5, graph=rng.random() < 0.5)
        c["F"] = rng.choice([2048, 3072, 4096])
        if B <= 4:
            c.update(steps=rng.choice([1, 4, 10] if B == 1 else [1, 2, 4]), m=rng.choice([0, 1, 1, 3]))
        return c
    if kind == "prefix":
        B = _log_int(rng, 1, 12)
        return dict(PREFIX, B=B, n=rng.randint(1, B), L=rng.randint(6, 18), S=_log_int(rng, 48, 1000), staged=rng.random() < 0.5)
    form = rng.choice(["batched", "long", "frames", "heads", "fp32"])
    if form == "batched":
        return dict(PATH, B=_log_int(rng, 1, 64), L=rng.randint(1, 4), S=rng.randint(200, 900), T=rng.randint(8, 64), ragged=rng.random() < 0.5,
                    m=rng.choice([0, 1, 5]), causal=rng.random() < 0.3)
    if form == "long":
        return dict(PATH, B=_log_int(rng, 1, 16), S=_log_int(rng, 1000, 4160), N=rng.choice([32, 100, 256]), outliers=True, ragged=rng.random() < 0.3)
    if form == "frames":
        B = _log_int(rng, 1, 16)
        return dict(PATH, B=B, N=256 * _log_int(rng, 1, max(1, min(50, 160 // B))), T=rng.randint(25, 100), m=256)
    if form == "heads":
        d = rng.choice([64, 128, 256])
        Hkv = rng.choice([1, 2, 4])
        return dict(PATH, B=_log_int(rng, 1, 16), L=rng.randint(1, 4), Hq=Hkv * rng.choice([2, 4, 8]), Hkv=Hkv, d=d, S=rng.randint(64, 600), ragged=rng.random() < 0.5,
                    N=rng.randint(16, 64), T=rng.randint(8, 64), D=rng.choice([512, 1024, 2048]), m=rng.choice([0, 1, 3]), causal=rng.random() < 0.5)
    return dict(PATH, dtype="f32", L=rng.randint(1, 2), Hq=rng.choice([2, 4]), d=64, S=rng.randint(32, 128), N=rng.randint(8, 32), T=rng.randint(4, 16), D=128, Cd=40,
                Hd=32, A=8, steps=rng.randint(1, 4), m=1)


# ---- inputs ------------------------------------------------------------------------------------------------------------

def _workload(c, seed):
    return synth.Workload(c["kind"], seed, synth.DTYPE_F32 if c["dtype"] == "f32" else synth.DTYPE_BF16, B=c["B"], L=c["L"], Hq=c["Hq"], Hkv=c["Hkv"], d=c["d"],
                          S=c["S"], S_max=c["S"], N=c["N"], T=c["T"], D=c["D"], Cd=c["Cd"], Hd=c["Hd"], A=c["A"], K=max(10, c["steps"]), m=c["m"])


def _lengths(c):
    """Prefix tokens of every stream: all S, or spread over the upper half of S."""
    return [c["S"] - (b * 37) % max(1, c["S"] // 2) if c["ragged"] else c["S"] for b in range(c["B"])]


class _Inputs:
    def __init__(self, dtype, seed):
        self.dtype = torch.float32 if dtype == "f32" else torch.bfloat16
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def __call__(self, *shape, std=1.0, dtype=None):
        t = torch.randn(*shape, generator=self.g, device=DEV, dtype=torch.float32)
        return (t * std if std != 1.0 else t).to(dtype or self.dtype)


def _cache(w, c, rnd):
    """A cache in the middle of a stream: prefixes written, ring full and wrapped at a different place for every stream."""
    cache = rb.Cache(w.L, w.B, w.Hq, w.Hkv, w.d, w.S, w.N, w.T, w.dtype, device=DEV, ring_head0=[(b * 11 + 5) % w.N for b in range(w.B)])
    S = _lengths(c)
    for b0 in range(0, w.B, 8):
        ids = list(range(b0, min(w.B, b0 + 8)))
        kv = [rnd(len(ids), w.L, w.S, w.Hkv, w.d) for _ in range(2)]
        rb.reflex_cache_init_static(cache, ids, kv[0], kv[1], S=[S[b] for b in ids])
        kv = [rnd(len(ids), w.L, w.N, w.Hkv, w.d) for _ in range(2)]
        rb.reflex_cache_append_sliding(cache, ids, kv[0], kv[1])
    return cache


def _conds(w, c, dtype):
    """The conditioning vectors of the steps' flow times."""
    return [torch.from_numpy(synth.cond_vectors(w, 1.0 - k / w.K)).to(DEV).to(dtype).contiguous() for k in range(c["steps"])]


def _prepare_expert(c, seed):
    w, rnd = _workload(c, seed), _Inputs(c["dtype"], seed)
    cache = _cache(w, c, rnd)
    s = dict(c=c, w=w, cache=cache, ids=list(range(w.B)), expert=ActionExpert(w, cache, random_weights_device(w, c["F"], DEV, seed), c["F"], DEV),
             cond=_conds(w, c, rnd.dtype), noise=rnd(w.B, w.T, w.A, dtype=torch.float32), a=torch.empty((w.B, w.T, w.A), dtype=torch.float32, device=DEV))
    if c["m"]:
        s["new"] = [rnd(w.B, w.L, c["m"], w.Hkv, w.d) for _ in range(2)]
    if c["graph"]:
        _expert_pass(s)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            _expert_pass(s)
    return s


def _expert_pass(s):
    if "new" in s:
        rb.reflex_cache_append_sliding(s["cache"], s["ids"], s["new"][0], s["new"][1])
    s["a"].copy_(s["noise"])
    for k, cond in enumerate(s["cond"]):
        s["expert"].step(s["a"], cond, k)


def _prepare_path(c, seed):
    w, rnd = _workload(c, seed), _Inputs(c["dtype"], seed)
    x = [rnd(w.B, w.T, w.D) for _ in range(w.L)]
    if c["outliers"]:
        x = [torch.where(torch.rand(t.shape, generator=rnd.g, device=DEV) < 1e-3, t * 1e3, t) for t in x]
    empty = lambda t: torch.empty_like(t)
    s = dict(c=c, w=w, cache=_cache(w, c, rnd), ids=list(range(w.B)), x=x, q=[rnd(w.B, w.T, w.Hq, w.d) for _ in range(w.L)],
             k=[rnd(w.B, w.T, w.Hkv, w.d) for _ in range(w.L)], v=[rnd(w.B, w.T, w.Hkv, w.d) for _ in range(w.L)], cond=_conds(w, c, rnd.dtype),
             W1=rnd(w.L, w.Hd, w.Cd, std=0.02), b1=rnd(w.L, w.Hd, std=0.1), W2=rnd(w.L, w.D, w.Hd, std=0.02), b2=rnd(w.L, w.D, std=0.1),
             gates=torch.empty((w.L * w.B * (w.D + w.Hd),), dtype=torch.float32, device=DEV), vel=rnd(w.B, w.T, w.A), noise=rnd(w.B, w.T, w.A, dtype=torch.float32))
    s.update(y=[empty(t) for t in s["x"]], out=[empty(t) for t in s["q"]], a=empty(s["noise"]))
    n = w.B * w.D
    s["gate"] = [s["gates"][l * n:(l + 1) * n].view(w.B, w.D) for l in range(w.L)]
    if c["m"]:
        s["new"] = [rnd(w.B, w.L, c["m"], w.Hkv, w.d) for _ in range(2)]
    return s


def _path_pass(s):
    c, w, cache = s["c"], s["w"], s["cache"]
    if "new" in s:
        rb.reflex_cache_append_sliding(cache, s["ids"], s["new"][0], s["new"][1])
    s["a"].copy_(s["noise"])
    for k, cond in enumerate(s["cond"]):
        rb.reflex_adarmsnorm_gate(cond, s["W1"], s["b1"], s["W2"], s["b2"], s["gates"])
        for l in range(w.L):
            rb.reflex_adarmsnorm(s["x"][l], s["y"][l], None, None, None, None, None, gate_buf=s["gate"][l])
            rb.reflex_partitioned_attention(cache, l, s["q"][l], s["k"][l], s["v"][l], s["out"][l], dyn_mask=int(c["causal"]))
        rb.reflex_flow_step(s["a"], s["vel"], None, k, w.K)


def _prepare_prefix(c, seed):
    rnd = _Inputs(c["dtype"], seed)
    cache = rb.Cache(c["L"], c["B"], 8 * c["Hkv"], c["Hkv"], c["d"], c["S"], c["N"], 50, rb.DTYPE_BF16, device=DEV, static_banks=2 if c["staged"] else 1)
    ids = list(range(c["B"] - c["n"], c["B"]))
    return dict(c=c, cache=cache, ids=ids, S=[c["S"] - (i * 5) % max(1, c["S"] // 8) for i in range(c["n"])],
                kv=[rnd(c["n"], c["L"], c["S"], c["Hkv"], c["d"]) for _ in range(2)])


def prepare(case, seed):
    return {"expert": _prepare_expert, "path": _prepare_path, "prefix": _prepare_prefix}[case["kind"]](case, seed)


# ---- one pass ----------------------------------------------------------------------------------------------------------

def run(state):
    c, cache = state["c"], state["cache"]
    if c["kind"] == "prefix":
        if c["staged"]:
            rb.reflex_cache_stage_static(cache, state["ids"], state["kv"][0], state["kv"][1], S=state["S"])
            rb.reflex_cache_commit_static(cache, state["ids"])
        else:
            rb.reflex_cache_init_static(cache, state["ids"], state["kv"][0], state["kv"][1], S=state["S"])
        return [cache.k_slab, cache.v_slab]
    if c["kind"] == "path":
        _path_pass(state)
        return state["y"] + state["out"] + [state["a"]] + ([cache.k_slab, cache.v_slab] if c["m"] else [])
    if "graph" in state:
        state["graph"].replay()
    else:
        _expert_pass(state)
    return [state["a"], state["expert"].vel, state["expert"].h] + ([cache.k_slab, cache.v_slab] if c["m"] else [])


# ---- what a pass cannot do without -------------------------------------------------------------------------------------

def work(case):
    c = case
    es = 4 if c["dtype"] == "f32" else 2
    if c["kind"] == "prefix":
        rows = sum(c["S"] - (i * 5) % max(1, c["S"] // 8) for i in range(c["n"]))
        return {"bytes": 2 * 2 * rows * c["L"] * c["Hkv"] * c["d"] * es, "flops": 0}
    B, L, T, D, A, Hd, Cd, steps = c["B"], c["L"], c["T"], c["D"], c["A"], c["Hd"], c["Cd"], c["steps"]
    nq, nkv = c["Hq"] * c["d"], c["Hkv"] * c["d"]
    keys = sum(_lengths(c)) + B * (c["N"] + T)
    attn = 4.0 * T * nq * keys * L
    cached = 2 * (keys - B * T) * nkv * es * L
    append = 2 * 2 * B * L * c["m"] * nkv * es
    chunk = 2 * B * T * A * 4
    if c["kind"] == "path":
        gate_w = L * (Hd * Cd + D * Hd + Hd + D) * es
        gate = 2.0 * B * L * (Hd * Cd + D * Hd)
        layer = L * B * T * (2 * D + 2 * nq + 2 * nkv) * es
        return {"bytes": append + steps * (cached + layer + gate_w + B * Cd * es + B * T * A * es) + chunk, "flops": steps * (attn + gate)}
    F, n_norm = c["F"], 2 * L + 1
    proj = L * (D * (nq + 2 * nkv) + nq * D + 3 * F * D) + 2 * A * D
    gate_w = n_norm * (Hd * Cd + D * Hd + Hd + D)
    return {"bytes": append + steps * (cached + (proj + gate_w) * es + B * Cd * es) + chunk,
            "flops": steps * (attn + 2.0 * B * T * proj + 2.0 * B * n_norm * (Hd * Cd + D * Hd))}


def tolerance(case):
    """Relative errors, about four times what was measured between the tensor-core kernels and the plain fp32-FMA kernels on the same
    inputs: attention and norm outputs 2.5e-3; a whole expert step 1.3e-2 on the residual stream and the velocity after 18 layers of
    bf16 activations (1.6e-2 after ten steps)."""
    if case["kind"] == "prefix":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": 5e-2 if case["kind"] == "expert" else 1e-2}
