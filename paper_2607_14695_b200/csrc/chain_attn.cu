// Partitioned attention (Eq. 1) for one or two streams: one launch, keys split over the eight CTAs of a cluster.
//
// What bounds a single stream is latency: 368 MFLOP and 0.9 MB of K/V per layer, spread over the chip, are a microsecond of work
// in a chain of dependent steps. The batched kernel's key split needs a second launch and 64-128 KB of fp32 partials per CTA through
// global memory: 12.4 us per layer inside an expert step (898 keys, 50 tokens, 8 heads). This kernel takes about 8.
//   - A CTA owns 32 (64) query rows -- (token, head of the group) pairs -- and one of eight slices of the keys, at most 128, so that its
//     partial O is 32 x 256 and goes to its seven peers through distributed shared memory.
//   - Seven slices divide the static prefix, the eighth holds ring slots and dynamic tokens. Static and ring keys are asked for before
//     the wait for the preceding kernel when the caller vouches for them (early: nothing in an expert step writes cache regions);
//     only Q and the dynamic tokens come after it.
//   - S = Q K^T with M = 64 (rows in lanes 0-15 of every lane quarter), read as 16x256b fragments: a thread holds two rows and the
//     row maximum is two shuffles. With 32 rows the two warps of a lane quarter take 64 keys each.
//   - O^T = V^T P^T with the head dimension as M (V as the MN-major A operand): a thread holds one column of O for all rows, so that
//     four rows of it are one 16-byte st.async and a warp's store is 512 contiguous bytes of the owner's inbox. CTA r of the cluster
//     owns an eighth of the rows: it receives the slices' unnormalised O and (m, l), counted on one mbarrier, and writes the merged
//     rows. The inbox reuses the K tile; every CTA tells its peers when its Q K^T is done with it.
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

constexpr int kCaSlices = 8;               // CTAs of a cluster
constexpr int kCaKeys = 128;               // keys of a slice at most
constexpr int kCaM = 64;                   // rows of the Q K^T MMA
constexpr int kCaThreads = 64 + 256;
constexpr int kCaHD = 256;
constexpr unsigned long long kCaWaitNs = 1000000000ull;

// ROWS: query rows -- (token, head of the KV head's group) pairs -- of a CTA at most, 32 or 64
template <int ROWS> struct CaSmem {
    static constexpr int OWN = ROWS / kCaSlices;                 // rows a CTA of the cluster merges: one or two quads
    static constexpr uint32_t Q_CHUNK = ROWS * 128;
    static constexpr uint32_t Q = 0;                             // 4 chunks of [ROWS][128 B] (the MMA reads kCaM rows: the rest is whatever follows)
    static constexpr uint32_t K = Q + 4 * Q_CHUNK;               // 4 chunks of [128 keys][128 B]; later the inbox [8 slices][OWN / 4 quads][256][4] fp32
    static constexpr uint32_t V = K + 4 * kCaKeys * 128;
    static constexpr uint32_t P = V + 4 * kCaKeys * 128;         // 2 chunks of [ROWS][64 keys]
    static constexpr uint32_t MX = P + 2 * ROWS * 128;           // [2 key halves][32 rows] row maxima
    static constexpr uint32_t ML = MX + 256;                     // [8 slices][OWN] (m, l, l of the second key half, -)
    static constexpr uint32_t WGT = ML + kCaSlices * OWN * 16;   // [8 slices][OWN] weights of the merge
    static constexpr uint32_t BAR = WGT + kCaSlices * OWN * 4;
    static constexpr uint32_t TOTAL = BAR + 128 + 1024;
    static_assert(kCaSlices * (OWN / 4) * kCaHD * 16 <= 4 * kCaKeys * 128, "inbox fits in the K tile");
    static_assert(TOTAL <= 227u * 1024u, "shared memory budget");
};
enum { CB_Q = 0, CB_K, CB_V, CB_S, CB_VREADY, CB_P, CB_O, CB_FREE, CB_INBOX, CB_COUNT };

#ifdef REFLEX_CG_TRACE
__device__ unsigned long long g_ca_trace[160 * 12];      // [CTA][event] of the last launch, ns
#define CA_TRACE(ev) do { if (blockIdx.y == 0) g_ca_trace[blockIdx.x * 12 + (ev)] = globaltimer_ns(); } while (0)
#else
#define CA_TRACE(ev) do { } while (0)
#endif

struct CaParams {
    const StreamState *state;
    __nv_bfloat16 *out;
    uint32_t *status;
    int B, Hq, Hkv, G, S_max, N, T, layer, ring_off;
    int box;             // rows of the static box
    int dyn_row;         // tile row of the first dynamic token in the last slice
    int early;
    int g_log2;
    int units, tt;       // tiles of a stream and KV head; tokens of a tile: ROWS / G
    float scale_log2;
    ChainPrefetch pf;
};

// lanes 0-15 of the warp's quarter, 64 columns: register 4 g + j of thread t is row t / 4 + (j & 2 ? 8 : 0), column 8 g + 2 (t % 4) + (j & 1)
__device__ __forceinline__ void ca_tmem_ld_16x256b(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// bits [lo, hi) of a 64-bit word
__device__ __forceinline__ uint64_t ca_bits(int lo, int hi)
{
    lo = max(lo, 0); hi = min(hi, 64);
    if (hi <= lo) return 0ull;
    return (hi >= 64 ? ~0ull : (1ull << hi) - 1ull) & ~((1ull << lo) - 1ull);
}

template <int ROWS>
__global__ void __cluster_dims__(kCaSlices, 1, 1) __launch_bounds__(kCaThreads, 1)
chain_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_ks, const __grid_constant__ CUtensorMap tm_vs,
                  const __grid_constant__ CUtensorMap tm_kr, const __grid_constant__ CUtensorMap tm_vr, const __grid_constant__ CUtensorMap tm_kd,
                  const __grid_constant__ CUtensorMap tm_vd, const CaParams p)
{
    using L = CaSmem<ROWS>;
    constexpr int OWN = L::OWN, QUADS = OWN / 4;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    auto bar = [&](int i) -> uint32_t { return base + L::BAR + 8u * (uint32_t)i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + L::BAR + 8 * CB_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int slice = (int)cluster_ctarank();
    const int unit = blockIdx.x >> 3, b = blockIdx.y;
    const int hkv = p.Hkv == 1 ? 0 : unit / p.units, t0 = (unit - hkv * p.units) * p.tt;   // KV head, first token
    const int rows = min(p.tt, p.T - t0) * p.G;                      // query rows of this CTA: (token, head in group)
    const int own = max(0, min(OWN, rows - slice * OWN));            // query rows this CTA merges
    const bool last = slice == kCaSlices - 1;                        // ring and dynamic tokens

    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (warp == 0) {
        if (lane == 0) {
            CA_TRACE(0);
            for (int i = 0; i < CB_COUNT; ++i) mbar_init(bar(i), i == CB_VREADY || i == CB_P ? 4u : i == CB_FREE ? (uint32_t)kCaSlices : 1u);
            *abort_flag = 0u;
            fence_mbar_init();
            mbar_expect_tx(bar(CB_INBOX), (uint32_t)(kCaSlices * (((own + 3) / 4) * kCaHD * 16 + own * (ROWS == 64 ? 8 : 12))));
        }
        __syncwarp();
        cluster_arrive();
        asm volatile("bar.arrive 4, %0;" ::"n"(kCaThreads) : "memory");
    } else {
        if (warp == 1) tmem_alloc(smem_u32((const void *)tmem_slot), 256);
        else if (warp == 2 && lane == 0) { prefetch_tmap(&tm_q); prefetch_tmap(&tm_kd); prefetch_tmap(&tm_vd); }
        __syncwarp();
        tc_fence_before();
        cluster_arrive();
    }
    // ---- geometry of the slice ----
    const StreamState ss = p.state[b];
    const int S = max(ss.static_len, 0), count = min(ss.count, p.N);
    const int row_base = (p.layer * p.B + b) * (p.ring_off + p.N);
    const int per = (S + kCaSlices - 2) / (kCaSlices - 1);
    const int k0 = slice * per;
    const int n_static = last ? 0 : max(0, min(per, S - k0));
    const int ext = last ? p.dyn_row + p.T : n_static;               // tile rows that may hold keys
    uint64_t live_lo, live_hi;
    if (last) {
        int oldest = ss.head - ss.count;                              // live ring slots: the circular run of `count` from here
        oldest %= p.N;
        if (oldest < 0) oldest += p.N;
        const int end = oldest + count;
        live_lo = ca_bits(oldest, min(end, p.N)) | (end > p.N ? ca_bits(0, end - p.N) : 0ull) | ca_bits(p.dyn_row, ext);
        live_hi = ca_bits(p.dyn_row - 64, ext - 64);
    } else {
        live_lo = ca_bits(0, ext);
        live_hi = ca_bits(-64, ext - 64);
    }
    // The producer goes from its barriers straight to its loads, the hand-shakes of block and cluster are the other warps' business: a CTA that
    // starts late, for lack of room beside the preceding kernel, has its first operands that much sooner.
    if (warp == 0) {
        // K and V of the cached regions (a whole box each; rows past the slice are masked)
        const uint32_t kv_bytes = last ? (uint32_t)((count > 0 ? p.N : 0) + p.T) * (kCaHD * 2) : n_static > 0 ? (uint32_t)p.box * (kCaHD * 2) : 0u;
        const bool some = last ? count > 0 : n_static > 0;
        const CUtensorMap *mk = last ? &tm_kr : &tm_ks, *mv = last ? &tm_vr : &tm_vs;
        const int r0 = row_base + (last ? p.ring_off : ss.bank * p.S_max + k0);
        mbar_expect_tx_elect(bar(CB_K), kv_bytes);
        if (some)
            for (int c = 0; c < 4; ++c) tma_load_3d_elect(base + L::K + c * (kCaKeys * 128), mk, bar(CB_K), c * 64, hkv, r0);
        mbar_expect_tx_elect(bar(CB_V), kv_bytes);
        if (some)
            for (int c = 0; c < 4; ++c) tma_load_3d_elect(base + L::V + c * (kCaKeys * 128), mv, bar(CB_V), c * 64, hkv, r0);
    } else {
        asm volatile("bar.sync 4, %0;" ::"n"(kCaThreads) : "memory");
        cluster_wait();              // the peers' barriers exist
        tc_fence_after();
    }
    if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    // (not before this CTA has its tensor memory: a dependent that took the columns first would wait for this grid, and this grid for them)
    if (warp != 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem = warp == 0 ? 0u : *tmem_slot;

    if (threadIdx.x == 0) CA_TRACE(1);
    auto wait_slow = [&](int i, uint32_t code) -> bool {
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t n = 1;; ++n) {
            if (mbar_try_wait_cluster(bar(i), 0)) return true;
            if ((n & 255u) == 0u) {
                if (*abort_flag) return false;
                if (globaltimer_ns() - t_start > kCaWaitNs) break;
            }
        }
        *abort_flag = 1u;
        if (p.status) atomicCAS(p.status, 0u, status_word(kSiteChainAttn + code));
        return false;
    };
    auto wait = [&](int i, uint32_t code) -> bool { return mbar_try_wait(bar(i), 0) || wait_slow(i, code); };
    auto wait_cl = [&](int i, uint32_t code) -> bool { return mbar_try_wait_cluster(bar(i), 0) || wait_slow(i, code); };

    if (warp == 0) {
        mbar_expect_tx_elect(bar(CB_Q), ROWS * kCaHD * 2);
        for (int c = 0; c < 4; ++c) tma_load_4d_elect(base + L::Q + c * L::Q_CHUNK, &tm_q, bar(CB_Q), c * 64, hkv * p.G, t0, b);
        if (last) {
            for (int c = 0; c < 4; ++c) tma_load_3d_elect(base + L::K + c * (kCaKeys * 128) + p.dyn_row * 128, &tm_kd, bar(CB_K), c * 64, hkv, b * p.T);
            for (int c = 0; c < 4; ++c) tma_load_3d_elect(base + L::V + c * (kCaKeys * 128) + p.dyn_row * 128, &tm_vd, bar(CB_V), c * 64, hkv, b * p.T);
        }
        cluster_wait();              // the peers' barriers exist
        if (lane == 0) {
            // this CTA's Q K^T is through with the K tile: its peers may send their partial results over it
            wait(CB_S, 1);
            for (int r = 0; r < kCaSlices; ++r)
                mbar_arrive_cluster_release(mapa(bar(CB_FREE), (uint32_t)r));
        }
        __syncwarp();
        chain_prefetch(p.pf, blockIdx.x + gridDim.x * blockIdx.y, gridDim.x * gridDim.y, lane);
    } else if (warp == 1) {
        constexpr uint32_t idesc_qk = umma_idesc_bf16(kCaM, kCaKeys, false);
        constexpr uint32_t idesc_pv = umma_idesc_bf16(128, ROWS, false) | (1u << 15);     // A is MN-major
        bool ok = wait(CB_K, 2) && wait(CB_Q, 3);
        if (lane == 0) CA_TRACE(2);
        if (ok && ext > 0) {
            tc_fence_after();
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint64_t ad = umma_desc_sw128(base + L::Q + c * L::Q_CHUNK, 16, 1024);
                uint64_t bd = umma_desc_sw128(base + L::K + c * (kCaKeys * 128), 16, 1024);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    umma_ss_elect(tmem, ad, bd, idesc_qk, (c > 0 || kk > 0) ? 1u : 0u);
                    umma_desc_advance(ad, 32);
                    umma_desc_advance(bd, 32);
                }
            }
        }
        umma_commit_elect(bar(CB_S));
        ok = ok && wait(CB_VREADY, 4) && wait(CB_P, 5);
        if (ok && ext > 0) {
            tc_fence_after();
            const int steps = (ext + 15) / 16;
            for (int kk = 0; kk < steps; ++kk) {
                const uint64_t bd = umma_desc_sw128(base + L::P + (kk >> 2) * (ROWS * 128) + (kk & 3) * 32, 16, 1024);
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    umma_ss_elect(tmem + 128 + h * ROWS, umma_desc_sw128(base + L::V + h * (2 * kCaKeys * 128) + kk * (16 * 128), kCaKeys * 128, 1024), bd, idesc_pv,
                                  kk > 0 ? 1u : 0u);
            }
        }
        umma_commit_elect(bar(CB_O));
    } else {
        const int t = threadIdx.x - 64, quarter = warp & 3, group = (warp - 2) >> 2;
        bool ok = true;
        // Four warps run the softmax, the other four clear V. 64 rows: warps of group 0, one lane quarter (16 rows) each, all 128
        // keys. 32 rows: they sit in lane quarters 0 and 1; the two warps of a quarter take 64 keys each.
        const bool softmax = ROWS == 64 ? group == 0 : quarter < 2;
        if (!softmax) {
            // V rows inside the contraction that hold no key: zero, so that weight 0 meets no stale NaN
            ok = wait(CB_V, 6);
            const int ext16 = (ext + 15) & ~15;
            uint64_t dead[2] = {~live_lo & ca_bits(0, ext16), ~live_hi & ca_bits(0, ext16 - 64)};
            const int chunk = ROWS == 64 ? quarter : (quarter & 1) + 2 * group;
            uint8_t *v = smem + L::V + chunk * (kCaKeys * 128) + lane * 4;
#pragma unroll
            for (int w = 0; w < 2; ++w)
                while (dead[w]) {
                    const int r = __ffsll((long long)dead[w]) - 1;
                    dead[w] &= dead[w] - 1;
                    *reinterpret_cast<uint32_t *>(v + (w * 64 + r) * 128) = 0u;
                }
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(CB_VREADY));
        } else {
            constexpr int NW = ROWS == 64 ? 2 : 1;      // 64-key halves per warp
            const int w0 = ROWS == 64 ? 0 : group;
            ok = wait(CB_S, 7);
            if (threadIdx.x == 64 + (ROWS == 64 ? 0 : 64)) CA_TRACE(3);
            tc_fence_after();
            uint32_t s[NW][32];
            const uint32_t addr = tmem + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
            for (int w = 0; w < NW; ++w) ca_tmem_ld_16x256b(addr + (w0 + w) * 64, s[w]);
            tmem_wait_ld();
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const uint64_t live = w0 + w == 0 ? live_lo : live_hi;
                if (live != ~0ull) {
                    const uint64_t ml = live >> (2 * (lane & 3));      // bit 8 g + j: this thread's column j of group g
#pragma unroll
                    for (int g = 0; g < 8; ++g)
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            if (!((ml >> (8 * g + j)) & 1ull)) { s[w][4 * g + j] = 0xff800000u; s[w][4 * g + 2 + j] = 0xff800000u; }
                }
            }
            float mrow[2];                            // the thread's two rows
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                float m = -INFINITY;
#pragma unroll
                for (int w = 0; w < NW; ++w)
#pragma unroll
                    for (int g = 0; g < 8; ++g) m = max3_f32(m, __uint_as_float(s[w][4 * g + 2 * hr]), __uint_as_float(s[w][4 * g + 2 * hr + 1]));
                m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
                mrow[hr] = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
            }
            if constexpr (ROWS == 32) {
                // the row's maximum over both halves of the keys
                float *mx = reinterpret_cast<float *>(smem + L::MX);
                const int r = quarter * 16 + (lane >> 2);
                if ((lane & 3) == 0) { mx[group * 32 + r] = mrow[0]; mx[group * 32 + r + 8] = mrow[1]; }
                asm volatile("bar.sync %0, 64;" ::"r"(2 + quarter) : "memory");
                mrow[0] = fmaxf(mrow[0], mx[(group ^ 1) * 32 + r]);
                mrow[1] = fmaxf(mrow[1], mx[(group ^ 1) * 32 + r + 8]);
            }
#pragma unroll
            for (int hr = 0; hr < 2; ++hr) {
                const float m = mrow[hr];
                const float ref = m == -INFINITY ? 0.f : -m * p.scale_log2;
                const int row = quarter * 16 + hr * 8 + (lane >> 2);
                uint8_t *pr = smem + L::P + w0 * (ROWS * 128) + row * 128 + (lane & 3) * 4;
                float l = 0.f;
#pragma unroll
                for (int w = 0; w < NW; ++w)
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        const float p0 = ex2(fmaf(__uint_as_float(s[w][4 * g + 2 * hr]), p.scale_log2, ref));
                        const float p1 = ex2(fmaf(__uint_as_float(s[w][4 * g + 2 * hr + 1]), p.scale_log2, ref));
                        l += p0 + p1;
                        __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
                        *reinterpret_cast<uint32_t *>(pr + w * (ROWS * 128) + ((g ^ (row & 7)) << 4)) = *reinterpret_cast<uint32_t *>(&pp);
                    }
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 2);
                if ((lane & 3) == 0 && row < rows) {
                    const uint32_t o = (uint32_t)(row / OWN), dst = mapa(base + L::ML + (uint32_t)(slice * OWN + row % OWN) * 16u, o), ib = mapa(bar(CB_INBOX), o);
                    if (ROWS == 64 || group == 0) st_async_v2(dst, ib, __float_as_uint(m * p.scale_log2), __float_as_uint(l));
                    else st_async_b32(dst + 8u, ib, __float_as_uint(l));
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(CB_P));
            if (threadIdx.x == 64 + (ROWS == 64 ? 0 : 64)) CA_TRACE(4);
        }
        // ---- partial O^T to the owners of the rows ----
        ok = wait(CB_O, 8) && ok;
        if (threadIdx.x == 64) CA_TRACE(5);
        tc_fence_after();
        const int d = group * 128 + quarter * 32 + lane;
        if (wait_cl(CB_FREE, 9)) {
#pragma unroll
            for (int c = 0; c < ROWS / 32; ++c) {
                if (ROWS == 32 || c * 32 < rows) {
                    uint32_t acc[32];
                    tmem_ld32(tmem + 128 + group * ROWS + ((uint32_t)(quarter * 32) << 16) + c * 32, acc);
                    tmem_wait_ld();
                    if (!ok || ext == 0) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[i] = ok ? 0u : 0x7fc00000u;
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int quad = c * 8 + q;
                        if (quad * 4 < rows) {
                            const uint32_t o = (uint32_t)(quad / QUADS);
                            st_async_v4(mapa(base + L::K + (uint32_t)((slice * QUADS + quad % QUADS) * kCaHD + d) * 16u, o), mapa(bar(CB_INBOX), o), acc[4 * q], acc[4 * q + 1],
                                           acc[4 * q + 2], acc[4 * q + 3]);
                        }
                    }
                }
            }
        }
        if (threadIdx.x == 64) CA_TRACE(6);
        tc_fence_before();
        // ---- merge of this CTA's rows ----
        if (own > 0) {
            ok = wait_cl(CB_INBOX, 10);              // (after a wait that ran out the rows are marked invalid, a quiet NaN, not left stale)
            if (threadIdx.x == 64) CA_TRACE(7);
            float *wgt = reinterpret_cast<float *>(smem + L::WGT);
            if (t < kCaSlices * OWN) {               // eight neighbouring lanes: the slices of one row
                const int r = t >> 3, q = t & 7;
                const float4 v = reinterpret_cast<const float4 *>(smem + L::ML)[q * OWN + r];
                float m = v.x;
                for (int o = 1; o < 8; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                const float w = v.x == -INFINITY ? 0.f : ex2(v.x - m);
                float l = w * (ROWS == 64 ? v.y : v.y + v.z);
                for (int o = 1; o < 8; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
                wgt[q * OWN + r] = w / l;
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
            const float4 *in = reinterpret_cast<const float4 *>(smem + L::K);
#pragma unroll
            for (int q2 = 0; q2 < QUADS; ++q2) {
                if (QUADS == 1 || q2 * 4 < own) {
                    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < kCaSlices; ++q) {
                        const float4 v = in[(q * QUADS + q2) * kCaHD + t];
                        const float4 w = *reinterpret_cast<const float4 *>(wgt + q * OWN + q2 * 4);
                        a.x = fmaf(v.x, w.x, a.x); a.y = fmaf(v.y, w.y, a.y); a.z = fmaf(v.z, w.z, a.z); a.w = fmaf(v.w, w.w, a.w);
                    }
                    const float o[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = slice * OWN + q2 * 4 + i, tk = r >> p.g_log2;
                        if (q2 * 4 + i < own) p.out[((size_t)(b * p.T + t0 + tk) * p.Hq + hkv * p.G + (r - (tk << p.g_log2))) * kCaHD + t] = __float2bfloat16_rn(ok ? o[i] : __int_as_float(0x7fc00000));
                    }
                }
            }
        }
    }
    if (threadIdx.x == 64) CA_TRACE(8);
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, 256);
    // Everything its peers send to a CTA has arrived before it leaves: their CB_FREE arrivals, their partial results. After a wait that
    // ran out that is not known: it stays until its peers' waits have run out as well.
    if (*abort_flag) {
        const unsigned long long ta = globaltimer_ns();
        while (globaltimer_ns() - ta < 6ull * kCaWaitNs) __nanosleep(1000);
    }
    if (threadIdx.x == 0) CA_TRACE(9);
}

}  // namespace

// Rows of a CTA: 32 while the clusters of eight fit the device at once, else 64 where the call stands by itself (0: too many streams). What a CTA
// sends through distributed shared memory is 1 KB per row at some 20 bytes per cycle. The device holds 15 clusters of eight (they need their SMs in
// one GPC); a cluster too many starts when another has finished.
// 64 rows would be faster as units of 128 (attn_pair.cuh): two streams x 382 keys 8.1 us against 10.6 here, x 898 keys 9.1 against 11.3. But the key
// that sets a slice's reference has weight 1, which bf16 holds exactly, and those have fewer slices and references than the eight here: 382 keys are
// 2.14e-3 from 64 bits there and 2.07e-3 here, 296 keys 2.26e-3 and 2.05e-3, 898 keys 2.13e-3 in both. Inside a step that distance does not
// show (layer output 3.46e-3 from 64 bits with either), so the units of 128 rows take it.
static int chain_attn_rows(const AttnParams &p, bool early)
{
    const int G = p.Hq / p.Hkv;
    for (int rows = 32; rows <= (early ? 32 : 64); rows *= 2) {
        if (rows % G != 0) continue;
        // On few keys the exchange of 64 rows costs more than the keys that the slices save (2 x 32 tokens x 112 keys 10.5 us, 8.8 by one CTA
        // per tile; 66 keys 9.3 and 8.0; from 313 keys on 0.92 to 1.02 of it; of 32 rows 0.6 to 1.0 everywhere).
        if (rows == 64 && p.S_max + p.N + p.T < 288) continue;
        const int tt = rows / G;
        if ((long long)p.B * p.Hkv * ((p.T + tt - 1) / tt) <= 14) return rows;
    }
    return 0;
}

bool chain_attn_supported(const AttnParams &p, bool early, int sm_count)
{
    if (p.dtype != REFLEX_DTYPE_BF16 || p.d != kCaHD || p.dyn_mask != 0 || sm_count < 148) return false;
    if (p.T > 64 || p.S_max > (kCaSlices - 1) * kCaKeys || (p.N + 7) / 8 * 8 + p.T > kCaKeys || p.N > 64) return false;
    return tc_supported(p) && chain_attn_rows(p, early) != 0;
}

template <typename K>
static cudaError_t launch_rows(K kernel, uint32_t smem, std::atomic<unsigned long long> &attr_set, const CUtensorMap *m, const CaParams &p, dim3 grid, cudaStream_t st)
{
    cudaError_t e = once_per_device(attr_set, [&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kCaThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, m[0], m[1], m[2], m[3], m[4], m[5], m[6], p);
    count_launch();
    return e;
}

cudaError_t launch_chain_attn(const AttnParams &a, uint32_t *status, bool early, const ChainPrefetch *pf, cudaStream_t st)
{
    const int rows = a.L * a.B * (a.ring_off + a.N);
    const int box = std::max(8, ((a.S_max + kCaSlices - 2) / (kCaSlices - 1) + 7) / 8 * 8);
    const int tile = chain_attn_rows(a, early), G = a.Hq / a.Hkv, tt = tile / G;
    CUtensorMap m[7];
    if (!tensor_map_q_bf16(&m[0], a.q, a.B, a.T, a.Hq, a.d, G, tt) || !tensor_map_kv_bf16(&m[1], a.k_slab, rows, a.Hkv, a.d, box) ||
        !tensor_map_kv_bf16(&m[2], a.v_slab, rows, a.Hkv, a.d, box) || !tensor_map_kv_bf16(&m[3], a.k_slab, rows, a.Hkv, a.d, a.N) ||
        !tensor_map_kv_bf16(&m[4], a.v_slab, rows, a.Hkv, a.d, a.N) || !tensor_map_kv_bf16(&m[5], a.k_dyn, a.B * a.T, a.Hkv, a.d, a.T) ||
        !tensor_map_kv_bf16(&m[6], a.v_dyn, a.B * a.T, a.Hkv, a.d, a.T))
        return cudaErrorInvalidValue;
    CaParams p;
    p.state = a.state; p.out = (__nv_bfloat16 *)a.out; p.status = status;
    p.B = a.B; p.Hq = a.Hq; p.Hkv = a.Hkv; p.G = G; p.S_max = a.S_max; p.N = a.N; p.T = a.T; p.layer = a.layer; p.ring_off = a.ring_off;
    p.box = box; p.dyn_row = (a.N + 7) / 8 * 8; p.early = early ? 1 : 0;
    p.g_log2 = 0;
    while ((1 << p.g_log2) < G) ++p.g_log2;      // (G divides 128: a power of two)
    p.units = (a.T + tt - 1) / tt; p.tt = tt;
    p.scale_log2 = a.scale * 1.4426950408889634f;
    p.pf = pf ? *pf : ChainPrefetch{};
    static std::atomic<unsigned long long> set32{0}, set64{0};
    const dim3 grid((unsigned)(kCaSlices * a.Hkv * p.units), (unsigned)a.B);
    return tile == 32 ? launch_rows(chain_attn_kernel<32>, CaSmem<32>::TOTAL, set32, m, p, grid, st) : launch_rows(chain_attn_kernel<64>, CaSmem<64>::TOTAL, set64, m, p, grid, st);
}

}  // namespace reflex

#ifdef REFLEX_CG_TRACE
extern "C" int reflex_debug_ca_trace(unsigned long long *out) { return (int)cudaMemcpyFromSymbol(out, reflex::g_ca_trace, sizeof(unsigned long long) * 160 * 12); }
#endif
