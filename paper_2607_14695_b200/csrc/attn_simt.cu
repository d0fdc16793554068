// Partitioned attention (Eq. 1), SIMT form: fp32 FMA, one warp per query row, online softmax over 32-key
// tiles, optional split over the key range with a merge of (m, l, acc) partials. Serves every supported
// shape and storage type; the tensor-core kernel takes over where the query tile is large enough.
//
// Keys are enumerated in one logical index space per stream:
//   [0, S)            static rows (S = static_len)
//   [S, S+N)          ring slots in PHYSICAL order; slot p is live iff ((p - (head-count)) mod N) < count
//   [S+N, S+N+T)      dynamic tokens, read in place from the caller's tensors
// Softmax does not depend on key order, so the ring is never unrolled or gathered.
#include <math.h>

#include "reflex_internal.cuh"

namespace reflex {

template <typename T, int DPL> struct RowIO;
template <int DPL> struct RowIO<__nv_bfloat16, DPL> {
    // lane-owned slice of DPL consecutive elements
    static __device__ __forceinline__ void load(const __nv_bfloat16 *p, float (&f)[DPL]) {
        if constexpr (DPL == 8) {
            uint4 u = *reinterpret_cast<const uint4 *>(p);
            const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
            for (int i = 0; i < 4; ++i) { float2 t = __bfloat1622float2(h[i]); f[2 * i] = t.x; f[2 * i + 1] = t.y; }
        } else {
#pragma unroll
            for (int i = 0; i < DPL; ++i) f[i] = __bfloat162float(p[i]);
        }
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, const float (&f)[DPL]) {
#pragma unroll
        for (int i = 0; i < DPL; ++i) p[i] = __float2bfloat16_rn(f[i]);
    }
};
template <int DPL> struct RowIO<float, DPL> {
    static __device__ __forceinline__ void load(const float *p, float (&f)[DPL]) {
        if constexpr (DPL % 4 == 0) {
#pragma unroll
            for (int i = 0; i < DPL; i += 4) { const float4 v = *reinterpret_cast<const float4 *>(p + i); f[i] = v.x; f[i + 1] = v.y; f[i + 2] = v.z; f[i + 3] = v.w; }
        } else {
#pragma unroll
            for (int i = 0; i < DPL; ++i) f[i] = p[i];
        }
    }
    static __device__ __forceinline__ void store(float *p, const float (&f)[DPL]) {
#pragma unroll
        for (int i = 0; i < DPL; ++i) p[i] = f[i];
    }
};

// Are a row's loads gathered before the first is used? In fp32 they are; in bf16, whose rows are half as many loads and have to be
// converted, the plain loops are the faster ones (32 rows x 976 keys, heads of 32: 20.6 us, 42.5 gathered), but for the widest heads with
// several warps per row (64 rows x 76 keys: 9.9 us, 8.1 gathered).
template <typename T, int DPL, int WPR> constexpr bool kSimtGather = sizeof(T) == 4 || (DPL == 8 && WPR > 1);

// dot of a K row (global, storage type) with a query row (shared, fp32), 8 elements per step; the loads of 64 elements in flight together
// where they are gathered
template <typename T, int D, bool GATHER>
__device__ __forceinline__ float dot_row(const T *__restrict__ k, const float *__restrict__ q_s)
{
    constexpr int CH = D < 64 ? D : 64;
    if constexpr (!GATHER) {
        float acc0 = 0.f, acc1 = 0.f;
        for (int e = 0; e < D; e += 8) {
            float f[8];
            RowIO<T, 8>::load(k + e, f);
            const float4 qa = *reinterpret_cast<const float4 *>(q_s + e), qb = *reinterpret_cast<const float4 *>(q_s + e + 4);
            acc0 = fmaf(f[0], qa.x, acc0); acc1 = fmaf(f[1], qa.y, acc1);
            acc0 = fmaf(f[2], qa.z, acc0); acc1 = fmaf(f[3], qa.w, acc1);
            acc0 = fmaf(f[4], qb.x, acc0); acc1 = fmaf(f[5], qb.y, acc1);
            acc0 = fmaf(f[6], qb.z, acc0); acc1 = fmaf(f[7], qb.w, acc1);
        }
        return acc0 + acc1;
    }
    float acc0 = 0.f, acc1 = 0.f;
#pragma unroll 1
    for (int e0 = 0; e0 < D; e0 += CH) {
        float f[CH / 8][8];
#pragma unroll
        for (int c = 0; c < CH / 8; ++c) RowIO<T, 8>::load(k + e0 + 8 * c, f[c]);
#pragma unroll
        for (int c = 0; c < CH / 8; ++c) {
            const float4 qa = *reinterpret_cast<const float4 *>(q_s + e0 + 8 * c);
            const float4 qb = *reinterpret_cast<const float4 *>(q_s + e0 + 8 * c + 4);
            acc0 = fmaf(f[c][0], qa.x, acc0); acc1 = fmaf(f[c][1], qa.y, acc1);
            acc0 = fmaf(f[c][2], qa.z, acc0); acc1 = fmaf(f[c][3], qa.w, acc1);
            acc0 = fmaf(f[c][4], qb.x, acc0); acc1 = fmaf(f[c][5], qb.y, acc1);
            acc0 = fmaf(f[c][6], qb.z, acc0); acc1 = fmaf(f[c][7], qb.w, acc1);
        }
    }
    return acc0 + acc1;
}

constexpr int kSimtWarps = 4;      // rows of a block, a warp each (WPR = 1)
constexpr int kSimtRowWarps = 8;   // warps that share a row (WPR = kSimtRowWarps)
// Does the grid take part in programmatic dependent launch? Not where many blocks run long: beside waiting blocks of the next grid they
// spread unevenly over the SMs (bf16, 2400 rows x 626 keys, heads of 256: 302 us, 438 with it).
template <typename T, int WPR> constexpr bool kSimtOverlap = WPR > 1 || sizeof(T) == 4;

// WPR: warps per query row. 1: a block takes kSimtWarps rows, grid = (ceil(T Hq / kSimtWarps), B, nsplit). kSimtRowWarps: a block
// takes one row, its warps every eighth tile of the slice, and merges their (m, l, acc) through shared memory, grid = (T Hq, B, nsplit).
// What bounds small problems is the latency of a tile, not the arithmetic: the rows of K and then batches of V rows are
// loaded with all loads in flight, and with few rows the tiles go to different warps (16 rows, 88 keys, fp32: 22.1 us with a warp
// per row, one load at a time and 3 tiles in a row).
template <typename T, int DPL, int WPR>
__global__ void __launch_bounds__(WPR == 1 ? kSimtWarps * 32 : WPR * 32)
attn_simt_kernel(AttnParams p)
{
    constexpr int d = DPL * 32;
    constexpr bool GATHER = kSimtGather<T, DPL, WPR>;
    constexpr int NB = DPL >= 8 ? 8 : DPL == 4 ? 16 : 32;      // V rows in flight
    __shared__ __align__(16) float q_s[WPR == 1 ? kSimtWarps : 1][d];
    if constexpr (kSimtOverlap<T, WPR>) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = blockIdx.y, split = blockIdx.z;
    const int rows = p.T * p.Hq;
    const int r = WPR == 1 ? blockIdx.x * kSimtWarps + warp : blockIdx.x;
    if (WPR == 1 && r >= rows) return;  // no block-wide barrier below
    const int t = r / p.Hq, h = r % p.Hq;
    const int kv = h / (p.Hq / p.Hkv);
    float *qs = q_s[WPR == 1 ? warp : 0];

    const T *q_row = (const T *)p.q + (((size_t)b * p.T + t) * p.Hq + h) * d;
    if (WPR == 1 || warp == 0) {
        float f[DPL];
        RowIO<T, DPL>::load(q_row + lane * DPL, f);
#pragma unroll
        for (int i = 0; i < DPL; ++i) qs[lane * DPL + i] = f[i];
    }
    const StreamState st = p.state[b];
    const int S = st.static_len > 0 ? st.static_len : 0;
    const int N = p.N;
    const int n_keys = S + N + p.T;
    const int n_tiles = (n_keys + 31) / 32;
    const int per = (n_tiles + p.nsplit - 1) / p.nsplit;
    const int tile0 = split * per;
    const int tile1 = min(n_tiles, tile0 + per);
    int oldest = (st.head - st.count) % N;  // physical slot of the oldest live token
    if (oldest < 0) oldest += N;

    const size_t row_elems = (size_t)p.Hkv * d;
    const size_t blk = ((size_t)p.layer * p.B + b) * (size_t)(p.ring_off + N);
    const size_t s_row0 = (size_t)st.bank * p.S_max;     // first row of the static bank in use
    const T *k_blk = (const T *)p.k_slab + blk * row_elems + (size_t)kv * d;
    const T *v_blk = (const T *)p.v_slab + blk * row_elems + (size_t)kv * d;
    const T *k_dyn = (const T *)p.k_dyn + (size_t)b * p.T * row_elems + (size_t)kv * d;
    const T *v_dyn = (const T *)p.v_dyn + (size_t)b * p.T * row_elems + (size_t)kv * d;
    if (WPR == 1) __syncwarp(); else __syncthreads();

    float m = -INFINITY, l = 0.f;
    float acc[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] = 0.f;

    for (int tile = tile0 + (WPR == 1 ? 0 : warp); tile < tile1; tile += WPR) {
        const int idx = tile * 32 + lane;
        const T *kp = nullptr, *vp = nullptr;
        if (idx < S) {
            kp = k_blk + (s_row0 + idx) * row_elems; vp = v_blk + (s_row0 + idx) * row_elems;
        } else if (idx < S + N) {
            const int slot = idx - S;
            int age = slot - oldest;
            if (age < 0) age += N;
            if (age < st.count) {
                kp = k_blk + (size_t)(p.ring_off + slot) * row_elems; vp = v_blk + (size_t)(p.ring_off + slot) * row_elems;
            }
        } else if (idx < n_keys) {
            const int j = idx - S - N;
            if (!(p.dyn_mask && j > t)) { kp = k_dyn + (size_t)j * row_elems; vp = v_dyn + (size_t)j * row_elems; }
        }
        const unsigned long long vaddr = (unsigned long long)vp;
        // a dead key's V row is never read (it may hold stale or poisoned bytes)
        float f[NB][DPL];
        auto load_v = [&](int j0) {
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const unsigned long long va = __shfl_sync(0xffffffffu, vaddr, j0 + j);
                if (va != 0ull) RowIO<T, DPL>::load((const T *)va + lane * DPL, f[j]);
                else {
#pragma unroll
                    for (int i = 0; i < DPL; ++i) f[j][i] = 0.f;
                }
            }
        };
        if constexpr (GATHER) load_v(0);
        float s = -INFINITY;
        if (kp) s = dot_row<T, d, GATHER>(kp, qs) * p.scale;
        float tmax = s;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
        const float m_new = fmaxf(m, tmax);
        if (m_new == -INFINITY) continue;  // nothing live so far (warp-uniform)
        const float alpha = (m == -INFINITY) ? 0.f : expf(m - m_new);
        const float pj = kp ? expf(s - m_new) : 0.f;
        float psum = pj;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, o);
        l = l * alpha + psum;
        m = m_new;
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[i] *= alpha;
        if constexpr (!GATHER) {
            for (int j = 0; j < 32; ++j) {
                const float w = __shfl_sync(0xffffffffu, pj, j);
                const unsigned long long va = __shfl_sync(0xffffffffu, vaddr, j);
                if (va == 0ull) continue;
                float v[DPL];
                RowIO<T, DPL>::load((const T *)va + lane * DPL, v);
#pragma unroll
                for (int i = 0; i < DPL; ++i) acc[i] = fmaf(w, v[i], acc[i]);
            }
        } else
#pragma unroll 1
        for (int j0 = 0; j0 < 32; j0 += NB) {
            if (j0 > 0) load_v(j0);
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const float w = __shfl_sync(0xffffffffu, pj, j0 + j);
#pragma unroll
                for (int i = 0; i < DPL; ++i) acc[i] = fmaf(w, f[j][i], acc[i]);
            }
        }
    }

    if constexpr (WPR > 1) {
        // the warps' partial results: warp 0 adds them up
        __shared__ float part[WPR][d + 2];
        part[warp][d] = m; part[warp][d + 1] = l;
#pragma unroll
        for (int i = 0; i < DPL; ++i) part[warp][lane * DPL + i] = acc[i];
        __syncthreads();
        if (warp > 0) return;
        const int live = min(WPR, tile1 - tile0);       // warps that had a tile
        for (int w = 1; w < live; ++w) m = fmaxf(m, part[w][d]);
        l = 0.f;
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
        for (int w = 0; w < live; ++w) {
            const float mw = part[w][d];
            if (mw == -INFINITY) continue;
            const float a = expf(mw - m);
            l = fmaf(part[w][d + 1], a, l);
#pragma unroll
            for (int i = 0; i < DPL; ++i) acc[i] = fmaf(part[w][lane * DPL + i], a, acc[i]);
        }
    }
    if (p.nsplit == 1) {
        const float inv = 1.f / l;  // l > 0: a dynamic query always sees itself
#pragma unroll
        for (int i = 0; i < DPL; ++i) acc[i] *= inv;
        T *o = (T *)p.out + (((size_t)b * p.T + t) * p.Hq + h) * d;
        RowIO<T, DPL>::store(o + lane * DPL, acc);
    } else {
        const size_t slot = partial_slot(b, rows, r, p.nsplit, split);
        float *po = partial_o(p.partials, slot, d), *pml = partial_ml(p.partials, (size_t)p.B * rows * p.nsplit, slot, d);
        if (lane == 0) { pml[0] = m; pml[1] = l; }
#pragma unroll
        for (int i = 0; i < DPL; ++i) po[lane * DPL + i] = acc[i];
    }
}

// Merge of split partials: m* = max m_s, l = sum l_s e^{m_s-m*}, o = sum acc_s e^{m_s-m*} / l. One warp per query row
// (lane s fetches slice s's (m, l); every lane owns d/32 output columns), 8 rows per block, all loads independent.
template <typename T, int DPL>
__global__ void __launch_bounds__(256)
attn_merge_kernel(AttnParams p)
{
    constexpr int d = DPL * 32;
    // launched with programmatic stream serialisation: wait for the attention kernel ahead of it before reading its partials
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = p.T * p.Hq;
    const int gr = blockIdx.x * 8 + warp;      // row over all streams
    if (gr >= p.B * rows) return;
    const int b = gr / rows, r = gr % rows;
    const size_t n_slots = (size_t)p.B * rows * p.nsplit;
    const size_t slot0 = partial_slot(b, rows, r, p.nsplit, 0);
    float ms = -INFINITY, ls = 0.f;
    if (lane < p.nsplit) {
        const float2 ml = *reinterpret_cast<const float2 *>(partial_ml(p.partials, n_slots, slot0 + lane, d));
        ms = ml.x; ls = ml.y;
    }
    float mstar = ms;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mstar = fmaxf(mstar, __shfl_xor_sync(0xffffffffu, mstar, o));
    const float w = (ms == -INFINITY) ? 0.f : expf(ms - mstar);
    float l = ls * w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    float acc[DPL];
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] = 0.f;
    // Slices in batches of eight: all of a batch's loads are issued before the first is used (guarded one by one, every slice
    // was an L2 round trip of its own in front of the next). An empty slice never wrote its O row: whatever is read there
    // is dropped by the weight test, not multiplied by zero.
    for (int s0 = 0; s0 < p.nsplit; s0 += 8) {
        float f[8][DPL], ws[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int s = min(s0 + j, p.nsplit - 1);
            ws[j] = s0 + j < p.nsplit ? __shfl_sync(0xffffffffu, w, s) : 0.f;
            const float *po = partial_o(p.partials, slot0 + s, d) + lane * DPL;
            if constexpr (DPL % 4 == 0) {
#pragma unroll
                for (int i = 0; i < DPL; i += 4) {
                    const float4 v = *reinterpret_cast<const float4 *>(po + i);
                    f[j][i] = v.x; f[j][i + 1] = v.y; f[j][i + 2] = v.z; f[j][i + 3] = v.w;
                }
            } else {
#pragma unroll
                for (int i = 0; i < DPL; ++i) f[j][i] = po[i];
            }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            if (ws[j] != 0.f) {
#pragma unroll
                for (int i = 0; i < DPL; ++i) acc[i] = fmaf(f[j][i], ws[j], acc[i]);
            }
        }
    }
    const float inv = 1.f / l;
#pragma unroll
    for (int i = 0; i < DPL; ++i) acc[i] *= inv;
    const int t = r / p.Hq, h = r % p.Hq;
    T *out = (T *)p.out + (((size_t)b * p.T + t) * p.Hq + h) * d;
    RowIO<T, DPL>::store(out + lane * DPL, acc);
}

// Few rows: a block per row, its eight warps share the keys. fp32: the line lies where warps with a row each would no longer leave SMs
// idle. bf16, whose tiles are cheaper: while a warp has hardly more than one tile of 32 keys and the blocks are few (24 rows x 81 keys,
// heads of 128: 17.2 -> 7.7 us; 512 x 80, heads of 256: 21.7 -> 13; but 384 x 380, heads of 256: 34 -> 48, and 4 x 825 18.3 -> 36, where
// key slices go to more blocks). A single tile leaves nothing to share (fp32, 1536 rows x 32 keys: 18.4 us, 23.1 with a block per row).
static bool simt_row_blocks(const AttnParams &p)
{
    const long long rows = (long long)p.T * p.Hq * p.B;
    const int n_tiles = (p.S_max + p.N + p.T + 31) / 32;
    if (p.dtype == REFLEX_DTYPE_F32) return rows <= (n_tiles < 2 ? 512 : 2048);
    return n_tiles >= 2 && (n_tiles <= kSimtRowWarps ? rows <= 512 : rows <= 128 && n_tiles <= kSimtRowWarps * 3 / 2);
}

int simt_choose_splits(const AttnParams &p, size_t partial_bytes, int sm_count)
{
    const int rows = p.T * p.Hq;
    const bool rb = simt_row_blocks(p);
    const int blocks = rb ? rows * p.B : ((rows + kSimtWarps - 1) / kSimtWarps) * p.B;
    const int n_tiles = (p.S_max + p.N + p.T + 31) / 32;
    int want = (4 * sm_count + blocks - 1) / blocks;  // aim at ~4 blocks per SM
    const int per = rb ? 2 * kSimtRowWarps : 2;       // at least two key tiles per split and warp
    if (want > n_tiles / per) want = n_tiles / per;
    if (want > kMaxSplits) want = kMaxSplits;
    const size_t per_split = (size_t)p.B * rows * (p.d + 2) * sizeof(float);
    if (per_split > 0 && (size_t)want * per_split > partial_bytes) want = (int)(partial_bytes / per_split);
    if (want < 1) want = 1;
    return want;
}

template <typename T, int DPL>
static cudaError_t launch_simt_d(const AttnParams &p, cudaStream_t st)
{
    const int rows = p.T * p.Hq;
    const bool rb = simt_row_blocks(p);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = rb ? dim3(rows, p.B, p.nsplit) : dim3((rows + kSimtWarps - 1) / kSimtWarps, p.B, p.nsplit);
    cfg.blockDim = dim3(32 * (rb ? kSimtRowWarps : kSimtWarps));
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (rb ? kSimtOverlap<T, kSimtRowWarps> : kSimtOverlap<T, 1>) ? 1 : 0;
    return rb ? cudaLaunchKernelEx(&cfg, attn_simt_kernel<T, DPL, kSimtRowWarps>, p) : cudaLaunchKernelEx(&cfg, attn_simt_kernel<T, DPL, 1>, p);
}

template <typename T>
static cudaError_t launch_simt_t(const AttnParams &p, cudaStream_t st)
{
    cudaError_t e;
    switch (p.d / 32) {
        case 1: e = launch_simt_d<T, 1>(p, st); break;
        case 2: e = launch_simt_d<T, 2>(p, st); break;
        case 4: e = launch_simt_d<T, 4>(p, st); break;
        case 8: e = launch_simt_d<T, 8>(p, st); break;
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    if (e != cudaSuccess || p.nsplit == 1) return e;
    return launch_attention_merge(p, st);
}

template <typename T>
static cudaError_t launch_merge_t(const AttnParams &p, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((p.B * p.T * p.Hq + 7) / 8);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    switch (p.d / 32) {
        case 1: e = cudaLaunchKernelEx(&cfg, attn_merge_kernel<T, 1>, p); break;
        case 2: e = cudaLaunchKernelEx(&cfg, attn_merge_kernel<T, 2>, p); break;
        case 4: e = cudaLaunchKernelEx(&cfg, attn_merge_kernel<T, 4>, p); break;
        case 8: e = cudaLaunchKernelEx(&cfg, attn_merge_kernel<T, 8>, p); break;
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return e;
}

cudaError_t launch_attention_merge(const AttnParams &p, cudaStream_t st)
{
    if (p.dtype == REFLEX_DTYPE_BF16) return launch_merge_t<__nv_bfloat16>(p, st);
    return launch_merge_t<float>(p, st);
}

cudaError_t launch_attention_simt(const AttnParams &p, cudaStream_t st)
{
    if (p.dtype == REFLEX_DTYPE_BF16) return launch_simt_t<__nv_bfloat16>(p, st);
    return launch_simt_t<float>(p, st);
}

}  // namespace reflex
