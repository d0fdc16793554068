"""Rules that every kernel keeps and no run can show reliably, checked on the sources."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_14695_b200", "csrc")


def _kernels():
    """(file: name, parameters, body) of every __global__ function; comments taken out."""
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\((?:[^()]|\([^()]*\))*\)\s*)*(\w+)\s*\(([^{]*?)\)\s*\{", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            out.append((f"{os.path.basename(path)}: {m.group(1)}", m.group(2), text[m.end():i]))
    return out


KERNELS = _kernels()


def test_kernels_are_found():
    names = {n.split(": ")[1] for n, _, _ in KERNELS}
    assert {"chain_attn_kernel", "attn_pair_kernel", "chain_gemm_kernel", "chain_in_kernel", "tile_gemm_kernel", "attn_tc2_kernel", "gate_kernel",
            "flow_step_kernel", "init_static_kernel", "linear_half_kernel", "linear_res_tc_kernel"} <= names


def test_attention_kernels_are_the_ones_a_call_can_reach():
    """(Clusters of four with 128 rows per CTA were left with groups of 128 heads of 256 inside a step, which refuses more than 12288 / 256 heads.)"""
    assert {n.split(": ")[1] for n, _, _ in KERNELS if re.search(r"(attn|attention)_?\w*kernel", n)} == {
        "attn_merge_kernel", "attn_pair_kernel", "attn_simt_kernel", "attn_tc2_kernel", "attn_tc_kernel", "chain_attn_kernel"}


@pytest.mark.parametrize("kernel", [k for k in KERNELS if "tmem_alloc" in k[2]], ids=lambda k: k[0])
def test_tensor_memory_is_taken_before_dependents_are_released(kernel):
    """A dependent grid may move in as soon as it is released. If it takes tensor memory that this grid has yet to take, the two wait
    for one another."""
    _, _, body = kernel
    assert body.index("tmem_alloc") < body.index("griddepcontrol.launch_dependents")


@pytest.mark.parametrize("kernel", [k for k in KERNELS if re.search(r"griddepcontrol\.wait|wait_then_release", k[2])], ids=lambda k: k[0])
def test_inputs_read_behind_the_wait_may_not_be_taken_for_constants(kernel):
    """A programmatically launched grid may run beside the one that writes its inputs. A const __restrict__ parameter promises that
    nobody writes it while the kernel runs, so its loads could be moved ahead of the wait. (The weights of the plain gate kernels, which
    wait_prior marks, are read ahead of it on purpose: the launch in front of them writes none.)"""
    _, params, _ = kernel
    bad = re.findall(r"const [^,]*__restrict__ (\w+)", params)
    assert not [b for b in bad if not ("wait_prior" in params and b in ("W", "bias"))], bad


PROJECTIONS = [k for k in KERNELS if k[0].split(":")[0] in ("tile_gemm.cu", "linear_half.cu", "linear_tc.cu", "qkv_tc.cu", "chain_gemm.cu", "gate_tc.cu") and "commit" in k[2]]


@pytest.mark.parametrize("kernel", PROJECTIONS, ids=lambda k: k[0])
def test_sums_are_announced_only_when_complete(kernel):
    """After a wait that ran out a contraction is not complete. The warps that read the accumulator (in a pair those of the other CTA, which sees nothing
    of the failed wait) may take it for complete only by the barrier that the last commit arrives on: no commit, no result but NaN."""
    commits = re.findall(r"([^;{}]*)\bumma2?_commit\w*\(bar\w*(?:\((?:S::)?(\w+))?", kernel[2])
    last = [before for before, name in commits if name.endswith("_ACC") or not name]
    assert last and all(re.search(r"if \(ok\)\s*$", b) for b in last), last


@pytest.mark.parametrize("kernel", PROJECTIONS, ids=lambda k: k[0])
def test_a_tile_of_a_failed_wait_is_written_as_nan(kernel):
    """A store that is left out keeps what the last call wrote: the result is written whatever the waits said, and is NaN where one ran out."""
    _, _, body = kernel
    assert "0x7fc00000" in body
    assert not re.search(r"if \([^()]*\bok && (?:m0|dst)|if \(!ok \|\| f >=", body)


def test_a_reported_wait_names_its_kernel():
    """The status word holds a number for every wait: kernels count theirs from bases of their own, far enough apart."""
    header = open(os.path.join(CSRC, "reflex_internal.cuh")).read()
    sites = {n: int(v) for n, v in re.findall(r"(kSite\w+) = (\d+)", header)}
    used = {}
    for name, _, body in KERNELS:
        assert len(re.findall(r"atomicCAS\((?:p\.)?status,", body)) == len(re.findall(r"atomicCAS\((?:p\.)?status, 0u, status_word\(kSite", body)), name
        for base in set(re.findall(r"status_word\((kSite\w+)", body)):
            last = max([int(c) for c in re.findall(r"\bwait(?:_slow|_cl)?\([^;]*?, (\d+)u?\)", body)] + [int(c) for c in re.findall(base + r" \+ (\d+)u", body)] + [0])
            used[base] = (name, last)
    assert len(used) == len({n for n, _ in used.values()}) == 12, used       # one base a kernel, no two kernels on one
    bases = sorted(sites[b] for b in used) + [sites["kSiteEnd"]]
    for base, (name, last) in used.items():
        assert sites[base] + last < min(b for b in bases if b > sites[base]), name
