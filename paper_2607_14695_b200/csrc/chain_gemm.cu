// The projections of a whole expert step for few rows (one or a few streams), chained kernel to kernel.
//
// A layer of one stream reads 34.6 MB of weights (5.3 us at the measured HBM rate) through five dependent launches that do
// almost no arithmetic: what bounds them is the latency from one kernel's last store to the next one's first result. Three
// things shorten that path here, all of them possible because one host call (reflex_expert_step) owns the whole chain:
//   - weights are asked for BEFORE the wait for the preceding kernel (griddepcontrol.wait). Nothing inside a step writes
//     weights, and a kernel of the chain only starts once its predecessor has passed its own wait, which the first kernel
//     of the step does only when everything ahead of the step is complete: the loads see what the caller wrote.
//   - the adaptive norm sits in the epilogue of the projection that PRODUCES the residual stream: it writes h, h * gamma of
//     the norm that follows (bf16) and the sums of squares of its columns, both from h before its rounding. The projection takes
//     h * gamma straight by TMA (no rewriting of operand tiles in shared memory) and applies 1 / RMS to its accumulator.
//   - with the contraction split over the CTAs of a cluster, a CTA pushes its partial sums into the shared memory of the CTA
//     that finishes the row (st.async, counted on that CTA's mbarrier): no cluster barrier between the last MMA and the
//     sum. (Staged in the own shared memory and fetched by the owner behind a cluster barrier, accumulator to end took
//     5.6-7 k of the kernels' 9-12 k cycles.)
// Measured (D = 1024, F = 4096, 18 layers, graph replay): one stream 744 -> 590 us per step, 1305 -> 637 called directly (one host call
// instead of ninety); two streams 850 -> 733.
// Tile: 64 or 128 weight rows as the A operand (cta_group::1), a group of 32, 64 or 128 activation rows as N. A thread then holds
// one feature of consecutive rows: four of them are one 16-byte store, and a warp's store is 512 contiguous bytes of the owner's
// inbox (activations as the A operand put 32 separate 16-byte pieces into every store: 1.7 us from accumulator to sum).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "chain.cuh"
#include "reflex_internal.cuh"
#include "sm100_ptx.cuh"

namespace reflex {

using namespace ptx;

namespace {

constexpr int kCgThreads = 64 + 256;      // producer warp, MMA warp, eight epilogue warps
constexpr uint32_t kCgMaxStages = 16;
constexpr uint32_t kCgBarBytes = 512;     // barriers, tensor-memory slot, abort flag
constexpr uint32_t kCgRsBytes = 512;      // 1 / RMS of the rows this CTA finishes
constexpr unsigned long long kCgWaitNs = 1000000000ull;

enum { CG_FULL = 0, CG_EMPTY = kCgMaxStages, CG_ACC = 2 * kCgMaxStages, CG_INBOX, CG_COUNT };

#ifdef REFLEX_CG_TRACE
__device__ unsigned long long g_cg_trace[256 * 160 * 8];      // [launch][CTA][event] of the last 256 launches, ns
static unsigned g_cg_seq = 0;
#define CG_TRACE(ev) do { if (blockIdx.y == 0 && blockIdx.x < 160) g_cg_trace[(p.seq % 256 * 160 + blockIdx.x) * 8 + (ev)] = globaltimer_ns(); } while (0)
#else
#define CG_TRACE(ev) do { } while (0)
#endif

struct CgParams {
#ifdef REFLEX_CG_TRACE
    unsigned seq;
#endif
    int M, R, B;                // rows, rows per stream, streams
    int NT;                     // rows of a group (grid y): 64 or 128
    int chunks, cps;            // 64-wide chunks of the contraction per CTA; chunks per stage and barrier
    int ksplit, ks_log2;        // CTAs of a cluster that share a tile
    int q_log2;                 // log2 of the row quads of a group that one CTA of the cluster finishes: (NT / 4) / ksplit
    int stages, x_rows;         // stage ring; rows of the x box
    int n_feat;                 // output features (SwiGLU: hidden features)
    int w_row0, w_up;           // first row of this layer in the stacked weights; SwiGLU: rows from a gate row to its up row
    const __nv_bfloat16 *res;   // CG_RES: residual (may be h)
    __nv_bfloat16 *h, *xg;      // CG_RES outputs [M][n_feat]; CG_SWIGLU, CG_OUT: h = output
    const float *gate;          // CG_RES: gamma of the norm that follows, [B][n_feat]
    float *ss_out;              // CG_RES: [M][slots_out] sums of squares of 32 columns of h each
    const float *ss_in;         // other modes: [M][slots_in]
    int slots_in, slots_out;
    float inv_D, eps;
    __nv_bfloat16 *q, *k, *v;   // CG_QKV
    int nq, nk;
    float *a;                   // CG_OUT: action chunk, a += dt * velocity
    float dt;
    uint32_t *status;
    ChainPrefetch pf;           // ranges asked into the L2 for the kernels that follow
};

__device__ __forceinline__ uint2 pack4_bf16(float a, float b, float c, float d)
{
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<uint32_t *>(&lo), *reinterpret_cast<uint32_t *>(&hi));
}

// sum over the 32 lanes of four values: lane l ends with the total of value l / 8 (six shuffles instead of twenty)
__device__ __forceinline__ float warp_sum4(float v0, float v1, float v2, float v3, int lane)
{
    const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
    const float a = (up16 ? v2 : v0) + __shfl_xor_sync(0xffffffffu, up16 ? v0 : v2, 16);
    const float b = (up16 ? v3 : v1) + __shfl_xor_sync(0xffffffffu, up16 ? v1 : v3, 16);
    float c = (up8 ? b : a) + __shfl_xor_sync(0xffffffffu, up8 ? a : b, 8);
    c += __shfl_xor_sync(0xffffffffu, c, 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    return c;
}

template <int MODE, int FT>
__global__ void __launch_bounds__(kCgThreads)
chain_gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w, const CgParams p)
{
    constexpr uint32_t W_TILE = FT * 128;         // FT weight rows x 64
    constexpr uint32_t QUAD = FT * 16;            // four rows of FT features, fp32
    constexpr int HF = MODE == CG_SWIGLU ? FT / 2 : FT;      // output features of a tile
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    const uint32_t x_tile = (uint32_t)p.x_rows * 128u;
    const uint32_t x_stage = x_tile * p.cps, w_stage = W_TILE * p.cps;
    const uint32_t off_x = 0, off_w = (uint32_t)p.stages * x_stage, off_in = off_w + (uint32_t)p.stages * w_stage;
    const uint32_t off_bar = off_in + ((uint32_t)p.ksplit << p.q_log2) * QUAD;
    auto bar = [&](int i) -> uint32_t { return base + off_bar + 8u * (uint32_t)i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + off_bar + 8 * CG_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    float *rsm = reinterpret_cast<float *>(smem + off_bar + kCgBarBytes);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int krank = p.ksplit > 1 ? (int)cluster_ctarank() : 0;
    const int tile = blockIdx.x >> p.ks_log2;
    const int n0 = tile * HF;                                     // first output feature of the tile
    const int row0 = blockIdx.y * p.NT;                           // first row of the group
    const int live = min(p.NT, p.M - row0);                       // rows of the group that exist
    const int live_quads = (live + 3) >> 2;
    const int own_q0 = krank << p.q_log2;                         // this CTA finishes row quads [own_q0, own_q0 + own_q) of the group
    const int own_q = max(0, min(1 << p.q_log2, live_quads - own_q0));
    // (No division by a runtime value on the way to a load: each costs a lone thread some 130 cycles, more than the load itself.)
    const int col_first = krank * p.chunks * 64;                  // first column of this CTA's slice of the contraction
    const int w_row = p.w_row0 + n0;
    const int steps = p.chunks / p.cps;
    const int head = min(steps, p.stages);

    auto load_w = [&](int s, int st) {
        for (int cc = 0; cc < p.cps; ++cc) {
            const int col = col_first + (st * p.cps + cc) * 64;
            const uint32_t dst = base + off_w + (uint32_t)s * w_stage + (uint32_t)cc * W_TILE;
            tma_load_2d_elect(dst, &tm_w, bar(CG_FULL + s), col, w_row);
            if (MODE == CG_SWIGLU) tma_load_2d_elect(dst + W_TILE / 2, &tm_w, bar(CG_FULL + s), col, w_row + p.w_up);
        }
    };
    auto load_x = [&](int s, int st) {
        for (int cc = 0; cc < p.cps; ++cc)
            tma_load_2d_elect(base + off_x + (uint32_t)s * x_stage + (uint32_t)cc * x_tile, &tm_x, bar(CG_FULL + s), col_first + (st * p.cps + cc) * 64, row0);
    };
    if (warp == 0) {
        if (lane == 0) {
            CG_TRACE(0);
            for (int s = 0; s < p.stages; ++s) {
                mbar_init(bar(CG_FULL + s), 1);
                mbar_init(bar(CG_EMPTY + s), 1);
            }
            mbar_init(bar(CG_ACC), 1);
            mbar_init(bar(CG_INBOX), 1);
            *abort_flag = 0u;
            fence_mbar_init();
            mbar_expect_tx(bar(CG_INBOX), (uint32_t)((p.ksplit - 1) * own_q) * QUAD);
        }
        __syncwarp();
        for (int s = 0; s < head; ++s) {
            mbar_expect_tx_elect(bar(CG_FULL + s), w_stage + x_stage);
            load_w(s, s);
        }
        // weights that the stages do not hold are asked into the L2
        for (int c = head * p.cps; c < p.chunks; ++c) {
            tma_prefetch_2d_elect(&tm_w, col_first + c * 64, w_row);
            if (MODE == CG_SWIGLU) tma_prefetch_2d_elect(&tm_w, col_first + c * 64, w_row + p.w_up);
        }
    }
    if (warp == 1) tmem_alloc(smem_u32((const void *)tmem_slot), p.NT);
    tc_fence_before();
    __syncthreads();
    if (p.ksplit > 1) { cluster_arrive(); cluster_wait(); }     // every inbox barrier of the cluster exists
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (threadIdx.x == 0) CG_TRACE(2);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    auto wait_slow = [&](int i, uint32_t parity, uint32_t code) -> bool {
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t n = 1;; ++n) {
            if (i == CG_INBOX ? mbar_try_wait_cluster(bar(i), parity) : mbar_try_wait(bar(i), parity)) return true;
            if ((n & 255u) == 0u) {
                if (*abort_flag) return false;
                if (globaltimer_ns() - t_start > kCgWaitNs) break;
            }
        }
        *abort_flag = 1u;
        if (p.status) atomicCAS(p.status, 0u, status_word(kSiteChainGemm + code));
        return false;
    };
    auto wait = [&](int i, uint32_t parity, uint32_t code) -> bool { return mbar_try_wait(bar(i), parity) || wait_slow(i, parity, code); };

    if (warp == 0) {
        for (int s = 0; s < head; ++s) load_x(s, s);
        int s = 0;
        uint32_t ph = 0;
        for (int st = head; st < steps; ++st) {
            if (!wait(CG_EMPTY + s, ph, 1)) break;
            mbar_expect_tx_elect(bar(CG_FULL + s), w_stage + x_stage);
            load_x(s, st);
            load_w(s, st);
            if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        chain_prefetch(p.pf, blockIdx.x + gridDim.x * blockIdx.y, gridDim.x * gridDim.y, lane);
    } else if (warp == 1) {
        const uint32_t idesc = umma_idesc_bf16(FT, 0, false) | ((uint32_t)(p.NT >> 3) << 17);
        int s = 0;
        uint32_t ph = 0, acc = 0;
        bool ok = true;
        for (int st = 0; st < steps; ++st) {
            ok = wait(CG_FULL + s, ph, 2);
            if (!ok) break;
            if (st == 0 && lane == 0) CG_TRACE(3);
            if (st == steps - 1 && lane == 0) CG_TRACE(1);
            tc_fence_after();
            for (int cc = 0; cc < p.cps; ++cc) {
                uint64_t ad = umma_desc_sw128(base + off_w + (uint32_t)s * w_stage + (uint32_t)cc * W_TILE, 16, 1024);
                uint64_t bd = umma_desc_sw128(base + off_x + (uint32_t)s * x_stage + (uint32_t)cc * x_tile, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    umma_ss_elect(tmem, ad, bd, idesc, acc);
                    acc = 1u;
                    umma_desc_advance(ad, 32);
                    umma_desc_advance(bd, 32);
                }
            }
            if (st + p.stages < steps) umma_commit_elect(bar(CG_EMPTY + s));
            if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        if (ok) umma_commit_elect(bar(CG_ACC));
    } else {
        const int t = threadIdx.x - 64, quarter = warp & 3, group = (warp - 2) >> 2;
        // ---- what finishing needs beside the sums, while the operands are on their way ----
        const int f = t % HF, fg = n0 + f;        // this thread's feature in every quad it finishes
        const int q_first = t / HF;
        constexpr int Q_STEP = 256 / HF;
        const bool f_ok = fg < p.n_feat;
        float res4[4] = {0.f, 0.f, 0.f, 0.f}, gate4[4] = {0.f, 0.f, 0.f, 0.f};
        auto load_res = [&](int q) {
            const int r = row0 + (own_q0 + q) * 4;
            int b = r / p.R, rb = r - b * p.R;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (q < own_q && f_ok && r + i < p.M) {
                    if (p.res) res4[i] = __bfloat162float(p.res[(size_t)(r + i) * p.n_feat + fg]);
                    gate4[i] = p.gate[(size_t)b * p.n_feat + fg];
                }
                if (++rb == p.R) { rb = 0; ++b; }
            }
        };
        if constexpr (MODE == CG_RES) {
            load_res(q_first);
        } else {
            // 1 / RMS of the rows this CTA finishes: eight threads per row
            for (int r = t >> 3; r < own_q * 4; r += 32) {
                const int rg = row0 + own_q0 * 4 + r;
                float ss = 0.f;
                if (rg < p.M)
                    for (int j = t & 7; j < p.slots_in; j += 8) ss += p.ss_in[(size_t)rg * p.slots_in + j];
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) ss += __shfl_xor_sync(0xFFu << (lane & 24), ss, o);
                if ((t & 7) == 0) rsm[r] = rsqrtf(ss * p.inv_D + p.eps);
            }
        }
        __nv_bfloat16 *dst = p.h + fg;            // row 0 of this feature's column
        int pitch = p.n_feat;
        if constexpr (MODE == CG_QKV) {
            if (fg < p.nq) { dst = p.q + fg; pitch = p.nq; }
            else if (fg < p.nq + p.nk) { dst = p.k + (fg - p.nq); pitch = p.nk; }
            else { dst = p.v + (fg - p.nq - p.nk); pitch = p.nk; }
        }

        bool ok = wait(CG_ACC, 0u, 3);
        if (t == 0) CG_TRACE(4);
        tc_fence_after();
        // ---- the accumulator (lane = weight row, column = row of x) to the CTAs that finish its rows ----
        const int wf = FT == 128 ? quarter * 32 + lane : quarter * 16 + lane;      // weight row of the tile (M = 64: lanes 0-15 of a quarter)
        const bool wf_ok = FT == 128 || lane < 16;
        const int q_mask = (1 << p.q_log2) - 1;
        for (int cb = 0; cb < p.NT / 32; ++cb) {
            const int col = group * (p.NT / 2) + cb * 16;
            if (col >= live) break;                                // (uniform)
            uint32_t acc[16];
            tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + col, acc);
            tmem_wait_ld();
            if (!ok) {
#pragma unroll
                for (int i = 0; i < 16; ++i) acc[i] = 0x7fc00000u;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int Q = col / 4 + i, owner = Q >> p.q_log2;
                const uint32_t slot = off_in + (uint32_t)((krank << p.q_log2) + (Q & q_mask)) * QUAD + (uint32_t)wf * 16u;
                if (Q < live_quads && wf_ok) {
                    if (owner == krank) *reinterpret_cast<uint4 *>(smem + slot) = make_uint4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
                    else st_async_v4(mapa(base + slot, (uint32_t)owner), mapa(bar(CG_INBOX), (uint32_t)owner), acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
                }
            }
        }
        tc_fence_before();
        asm volatile("bar.sync 1, 256;" ::: "memory");             // rsm and this CTA's own share
        if (p.ksplit > 1 && own_q > 0) ok = (mbar_try_wait_cluster(bar(CG_INBOX), 0u) || wait_slow(CG_INBOX, 0u, 4)) && ok;
        if (t == 0) CG_TRACE(5);

        // ---- finish: one feature of four rows per thread and round ----
        for (int q = q_first; q < own_q; q += Q_STEP) {
            const uint8_t *src = smem + off_in + (uint32_t)q * QUAD + (uint32_t)f * 16u;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f), u = s;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if (k < p.ksplit) {
                    const float4 v = *reinterpret_cast<const float4 *>(src + (((uint32_t)k << p.q_log2) * QUAD));
                    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
                    if constexpr (MODE == CG_SWIGLU) {
                        const float4 w = *reinterpret_cast<const float4 *>(src + (((uint32_t)k << p.q_log2) * QUAD) + HF * 16);
                        u.x += w.x; u.y += w.y; u.z += w.z; u.w += w.w;
                    }
                }
            }
            float val[4] = {s.x, s.y, s.z, s.w};
            if (!ok) val[0] = val[1] = val[2] = val[3] = __int_as_float(0x7fc00000);      // a wait ran out: sums may be missing
            const int r = row0 + (own_q0 + q) * 4;
            if constexpr (MODE == CG_RES) {
                if (q != q_first) load_res(q);
                float sq[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sq[i] = 0.f;
                    if (f_ok && r + i < p.M) {
                        const float h = val[i] + res4[i];           // (the norm takes the sum before its rounding: one rounding less)
                        const size_t o = (size_t)(r + i) * p.n_feat + fg;
                        p.h[o] = __float2bfloat16_rn(h);
                        p.xg[o] = __float2bfloat16_rn(h * gate4[i]);
                        sq[i] = h * h;
                    }
                }
                const float tot = warp_sum4(sq[0], sq[1], sq[2], sq[3], lane);
                // lanes 0, 8, 16, 24 hold the sums of rows 0, 1, 2, 3 of the quad. (The width is a multiple of 64: with tiles of 128 features the
                // upper two warps of the last one may be past its end, and what would be their slots are the next row's.)
                if ((lane & 7) == 0 && f_ok && r + (lane >> 3) < p.M) p.ss_out[(size_t)(r + (lane >> 3)) * p.slots_out + (fg >> 5)] = tot;
            } else {
                const float4 rs = *reinterpret_cast<const float4 *>(rsm + q * 4);
                const float rs4[4] = {rs.x, rs.y, rs.z, rs.w}, uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float o = val[i] * rs4[i];
                    if constexpr (MODE == CG_SWIGLU) o = silu_mul(o, uu[i] * rs4[i]);
                    if (f_ok && r + i < p.M) {
                        const __nv_bfloat16 ov = __float2bfloat16_rn(o);
                        dst[(size_t)(r + i) * pitch] = ov;
                        if constexpr (MODE == CG_OUT) {             // the update takes the velocity as stored
                            float *a = p.a + (size_t)(r + i) * p.n_feat + fg;
                            *a = fmaf(p.dt, __bfloat162float(ov), *a);
                        }
                    }
                }
            }
        }
    }
    __syncwarp();
    if (threadIdx.x == 64) CG_TRACE(6);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, p.NT);
    // Everything its peers send to a CTA has arrived (CG_INBOX) before it leaves. After a wait that ran out that is not known: it
    // stays until its peers' waits have run out as well.
    if (p.ksplit > 1 && *abort_flag) {
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 4ull * kCgWaitNs) __nanosleep(1000);
    }
    if (threadIdx.x == 0) CG_TRACE(7);
}

struct CgConfig { int FT, NT, ksplit, cps, stages; };

constexpr uint32_t kCgSmemMax = 227u * 1024u;
// Rows up to which the chain is taken: a whole step of 1 / 2 / 3 / 4 streams of 50 tokens takes 595 / 733 / 955 / 980 us chained and
// 744 / 850 / 890 / 921 through the single calls, whose tiles then share the weights among more rows.
constexpr int kCgMaxRows = 128;

uint32_t cg_fixed(int FT, int NT) { return (uint32_t)(NT / 4) * FT * 16u + kCgBarBytes + kCgRsBytes + 1024u; }     // inbox, barriers, alignment

// The tile shape of a projection: among the shapes whose CTAs all fit the SMs at once, the one with the least estimated time.
bool cg_choose(int mode, int M, int K, int N, CgConfig &best)
{
    const int all_chunks = (K + 63) / 64;
    const int cols = mode == CG_SWIGLU ? 2 * N : N;
    double best_cost = 1e30;
    for (int NT = 32; NT <= 128; NT *= 2) {
        if (NT > 32 && M <= NT / 2) break;
        const int rows = std::min(NT, M), groups = (M + NT - 1) / NT, x_rows = (rows + 7) / 8 * 8;
        for (int FT = 64; FT <= 128; FT += 64) {
            if (mode == CG_SWIGLU && N % (FT / 2) != 0) continue;
            const int tiles = (cols + FT - 1) / FT;
            for (int ks = 1; ks <= 8; ks *= 2) {
                if (all_chunks % ks != 0 || NT / 4 < ks) continue;
                const int chunks = all_chunks / ks;
                // clusters of 8 and of 4 need their SMs in one GPC: the device holds 15 and 33 at once (1 CTA per SM), and a cluster too
                // many starts when another has finished
                if (tiles * groups * ks > 148 || (ks == 8 && tiles * groups > 14) || (ks == 4 && tiles * groups > 32)) continue;
                const int cps = chunks % 2 == 0 ? 2 : 1;
                const uint32_t stage = (uint32_t)(x_rows + FT) * 128u * cps, fixed = cg_fixed(FT, NT);
                const int steps = chunks / cps;
                if (fixed + stage * std::min(steps, 2) > kCgSmemMax) continue;
                const CgConfig c = {FT, NT, ks, cps, (int)std::min<uint32_t>({(uint32_t)steps, (kCgSmemMax - fixed) / stage, kCgMaxStages})};
                // Cycles, fitted to a sweep of all shapes at 50 and 100 rows (D = 1024, F = 4096): an SM takes in about 60 bytes per cycle
                // after the wait (all of x, the weights that the stages do not hold, and three tenths of those that they do); partial sums
                // cross the cluster at about 24; a finishing round takes some 200; weights that several row groups read count again.
                const double resident = (double)c.stages * cps * FT * 128, w = chunks * (double)FT * 128;
                const double ingest = (chunks * (double)x_rows * 128 + w - 0.7 * resident) / 60.0;
                const double mma = chunks * 4.0 * std::max((FT + NT) * 32 / 128.0, FT * NT / 256.0);
                const double push = ks > 1 ? 400.0 + rows * (double)FT * 4 * (ks - 1) / ks / 24.0 : 0.0;
                const double fin = (rows + 3) / 4 * (double)(mode == CG_SWIGLU ? FT / 2 : FT) / ks / 256.0 * 200.0;
                const double cost = std::max(ingest, mma) + 0.3 * std::min(ingest, mma) + push + fin + groups * (double)cols * K * 2 / 6000.0;
                if (cost < best_cost) { best_cost = cost; best = c; }
            }
        }
    }
    return best_cost < 1e30;
}

template <int MODE, int FT>
cudaError_t cg_launch(const CgConfig &c, const CUtensorMap &mx, const CUtensorMap &mw, const CgParams &p, dim3 grid, uint32_t smem, cudaStream_t st)
{
    static std::atomic<unsigned long long> attr_set{0};
    cudaError_t e0 = once_per_device(attr_set, [] { return cudaFuncSetAttribute(chain_gemm_kernel<MODE, FT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCgSmemMax); });
    if (e0 != cudaSuccess) return e0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kCgThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)c.ksplit; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = c.ksplit > 1 ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, chain_gemm_kernel<MODE, FT>, mx, mw, p);
    count_launch();
    return e;
}

template <int FT>
cudaError_t cg_launch_mode(int mode, const CgConfig &c, const CUtensorMap &mx, const CUtensorMap &mw, const CgParams &p, dim3 grid, uint32_t smem, cudaStream_t st)
{
    switch (mode) {
        case CG_RES: return cg_launch<CG_RES, FT>(c, mx, mw, p, grid, smem, st);
        case CG_QKV: return cg_launch<CG_QKV, FT>(c, mx, mw, p, grid, smem, st);
        case CG_SWIGLU: return cg_launch<CG_SWIGLU, FT>(c, mx, mw, p, grid, smem, st);
        default: return cg_launch<CG_OUT, FT>(c, mx, mw, p, grid, smem, st);
    }
}

}  // namespace

bool chain_proj_supported(int mode, int M, int K, int N)
{
    CgConfig c;
    return M >= 1 && K >= 8 && N >= 8 && (M <= kCgMaxRows || mode == CG_OUT) && K % 8 == 0 && N % 8 == 0 && cg_choose(mode, M, K, N, c);
}

cudaError_t launch_chain_proj(const ChainProj &a, cudaStream_t st)
{
    CgConfig c;
    const int M = a.B * a.R;
    if (!cg_choose(a.mode, M, a.K, a.N, c)) return cudaErrorInvalidValue;
    const int x_rows = (std::min(c.NT, M) + 7) / 8 * 8;
    const bool swiglu = a.mode == CG_SWIGLU;
    CUtensorMap mx, mw;
    if (!tensor_map_2d_bf16(&mx, a.x, a.K, M, x_rows) || !tensor_map_2d_bf16(&mw, a.W, a.K, a.w_rows, swiglu ? c.FT / 2 : c.FT)) return cudaErrorInvalidValue;
    auto log2i = [](int v) { int l = 0; while ((1 << l) < v) ++l; return l; };
    CgParams p = {};
    p.M = M; p.R = a.R; p.B = a.B; p.NT = c.NT; p.chunks = (a.K + 63) / 64 / c.ksplit; p.cps = c.cps; p.ksplit = c.ksplit; p.ks_log2 = log2i(c.ksplit);
    p.q_log2 = log2i(c.NT / 4 / c.ksplit); p.stages = c.stages; p.x_rows = x_rows;
    p.n_feat = a.N; p.w_row0 = a.w_row0; p.w_up = swiglu ? a.N : 0;
    p.res = a.res; p.h = a.h; p.xg = a.xg; p.gate = a.gate; p.ss_out = a.ss_out; p.ss_in = a.ss_in; p.slots_in = a.slots_in; p.slots_out = (a.N + 31) / 32;
    p.inv_D = a.D > 0 ? 1.f / (float)a.D : 0.f; p.eps = a.eps; p.q = a.q; p.k = a.k; p.v = a.v; p.nq = a.nq; p.nk = a.nk; p.a = a.a; p.dt = a.dt; p.status = a.status;
    p.pf = a.pf;
#ifdef REFLEX_CG_TRACE
    p.seq = g_cg_seq++;
#endif
    const int tiles = ((swiglu ? 2 * a.N : a.N) + c.FT - 1) / c.FT;
    const dim3 grid((unsigned)(tiles * c.ksplit), (unsigned)((M + c.NT - 1) / c.NT));
    const uint32_t smem = (uint32_t)(c.stages * c.cps * (x_rows + c.FT) * 128) + cg_fixed(c.FT, c.NT);
    return c.FT == 64 ? cg_launch_mode<64>(a.mode, c, mx, mw, p, grid, smem, st) : cg_launch_mode<128>(a.mode, c, mx, mw, p, grid, smem, st);
}

// ---- head of the step: the action chunk to tokens --------------------------------------------------------------------------
namespace {

constexpr int kCiRows = 4;       // rows at a time

// h = bf16(a) W_in^T with a contraction of A <= 32: fp32 FMAs, four features per thread, their weights in registers for all the row groups
// of the block; the block holds whole rows, so it finishes their sums of squares. (One group per block read the 64 KB of weights once
// for every four rows: 27 us for 3200 rows.)
template <int A>
__global__ void __launch_bounds__(256)
chain_in_kernel(const float *a, const __nv_bfloat16 *W, const float *gate, __nv_bfloat16 *h, __nv_bfloat16 *xg, float *ss_out, int M, int R, int D,
                int groups)
{
    __shared__ __align__(16) float as[kCiRows][A];
    __shared__ float part[kCiRows][8];
    uint4 w[4][A / 8];                                 // features f .. f + 3 of the first 1024
    const int f0 = threadIdx.x * 4;
    auto load_w = [&](int f) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k8 = 0; k8 < A / 8; ++k8) w[j][k8] = f < D ? *reinterpret_cast<const uint4 *>(W + (size_t)(f + j) * A + k8 * 8) : make_uint4(0u, 0u, 0u, 0u);
    };
    load_w(f0);                                        // (weights: nothing in a step writes them)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#pragma unroll 1
    for (int g = 0; g < groups; ++g) {
        const int row0 = (blockIdx.x * groups + g) * kCiRows;
        if (row0 >= M) break;
        for (int i = threadIdx.x; i < kCiRows * A; i += 256) {
            const int r = row0 + i / A;
            as[i / A][i % A] = r < M ? __bfloat162float(__float2bfloat16_rn(a[(size_t)r * A + i % A])) : 0.f;
        }
        __syncthreads();
#pragma unroll 1
        for (int fb = 0; fb < D; fb += 1024) {
            const int f = fb + f0;
            if (D > 1024) load_w(f);
#pragma unroll 1
            for (int r = 0; r < kCiRows; ++r) {
                float ss = 0.f;
                if (f < D && row0 + r < M) {
                    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int k8 = 0; k8 < A / 8; ++k8) {
                        const float4 a0 = *reinterpret_cast<const float4 *>(&as[r][k8 * 8]), a1 = *reinterpret_cast<const float4 *>(&as[r][k8 * 8 + 4]);
                        const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint32_t ww[4] = {w[j][k8].x, w[j][k8].y, w[j][k8].z, w[j][k8].w};
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                acc[j] = fmaf(av[2 * i + 1], __uint_as_float(ww[i] & 0xFFFF0000u), fmaf(av[2 * i], __uint_as_float(ww[i] << 16), acc[j]));
                        }
                    }
                    const float4 g4 = *reinterpret_cast<const float4 *>(gate + (size_t)((row0 + r) / R) * D + f);
                    const size_t o = (size_t)(row0 + r) * D + f;
                    *reinterpret_cast<uint2 *>(h + o) = pack4_bf16(acc[0], acc[1], acc[2], acc[3]);
                    *reinterpret_cast<uint2 *>(xg + o) = pack4_bf16(acc[0] * g4.x, acc[1] * g4.y, acc[2] * g4.z, acc[3] * g4.w);
                    ss = fmaf(acc[0], acc[0], fmaf(acc[1], acc[1], fmaf(acc[2], acc[2], acc[3] * acc[3])));
                }
                for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
                if ((threadIdx.x & 31) == 0) part[r][threadIdx.x >> 5] = fb == 0 ? ss : part[r][threadIdx.x >> 5] + ss;
            }
        }
        __syncthreads();
        if (threadIdx.x < kCiRows && row0 + (int)threadIdx.x < M) {
            float s = 0.f;
            for (int x = 0; x < 8; ++x) s += part[threadIdx.x][x];
            ss_out[row0 + threadIdx.x] = s;
        }
    }
}

}  // namespace

cudaError_t launch_chain_in(const float *a, const __nv_bfloat16 *W_in, const float *gate, __nv_bfloat16 *h, __nv_bfloat16 *xg, float *ss_out, int B,
                            int R, int D, int A, cudaStream_t st)
{
    const int M = B * R;
    cudaLaunchConfig_t cfg = {};
    const int all = (M + kCiRows - 1) / kCiRows, groups = (all + 295) / 296;       // about two blocks per SM
    cfg.gridDim = dim3((unsigned)((all + groups - 1) / groups));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    switch (A) {
        case 8: e = cudaLaunchKernelEx(&cfg, chain_in_kernel<8>, a, W_in, gate, h, xg, ss_out, M, R, D, groups); break;
        case 16: e = cudaLaunchKernelEx(&cfg, chain_in_kernel<16>, a, W_in, gate, h, xg, ss_out, M, R, D, groups); break;
        case 32: e = cudaLaunchKernelEx(&cfg, chain_in_kernel<32>, a, W_in, gate, h, xg, ss_out, M, R, D, groups); break;
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    return e;
}

}  // namespace reflex

#ifdef REFLEX_CG_TRACE
extern "C" int reflex_debug_cg_trace(unsigned long long *out, unsigned *seq)
{
    *seq = reflex::g_cg_seq;
    return (int)cudaMemcpyFromSymbol(out, reflex::g_cg_trace, sizeof(unsigned long long) * 256 * 160 * 8);
}
#endif

