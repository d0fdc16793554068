// The wide projections of an expert step for many rows: packed Q/K/V and the gate / up pair of the SwiGLU block, on operands that are
// ready as they lie. The residual projection in front writes h * gamma of the norm that follows and the rows' sums of squares
// (linear_tc.cu), so that nothing has to rewrite operand tiles here: out = epilogue((1 / RMS(h_r)) (h * gamma)_r . W^T).
//
// A CTA pair (cta_group::2) owns 256 rows x BN accumulator columns and walks its tiles; both operands come by TMA through a ring of
// 64-column stages. Two accumulators take turns, so that eight warps scale, convert and store one tile while the tensor pipe works on
// the next. For SwiGLU the B operand's two halves, one per CTA, are BN / 2 rows of W_gate and the same rows of W_up.
// What bounds it: a 256 x 256 step of 512 tensor cycles takes about 660, as it does in the library's GEMMs, with 32 KB a step
// and SM from the L2; at 300-800 rows the fixed part of a launch (first loads, last epilogue).
// Measured inside an expert step against the kernels that gate x in shared memory (D = 1024, F = 4096): gate/up 43.5 -> 34.4 us at 3200
// rows and 15.6 -> 10.0 at 429, Q/K/V 16.5 -> 15.1 and 7.6 -> 6.6; the residual projections in front pay 1.5 to 2.3 us each for h * gamma.
// At a few hundred rows a launch lasts as long as one CTA takes to take its operands in, at 50 to 58 bytes per cycle: pair tiles of 128 rows
// (BM = 64) where they lower that (tg_shape). Expert steps of 150 rows 770 -> 761 us, 200 rows 775 -> 770, 300 rows (F = 3072) 815 -> 789.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "chain.cuh"
#include "reflex_internal.cuh"
#include "sm100_ptx.cuh"

namespace reflex {

using namespace ptx;

namespace {

constexpr int kTgThreads = 64 + 256;      // producer warp, MMA warp, eight epilogue warps (two threads per row)
constexpr int kTgBK = 64;
constexpr unsigned long long kTgWaitNs = 1000000000ull;

template <int BN, int BM>
struct TgSmem {
    static constexpr int NST = BM == 64 ? (BN == 256 ? 7 : BN == 128 ? 10 : 13) : BN == 256 ? 5 : 6;
    static constexpr uint32_t A_STAGE = BM * 128;
    static constexpr uint32_t B_STAGE = (BN / 2) * 128;
    static constexpr uint32_t CHUNK = BM * 128;                   // BM rows x 64 output columns
    static constexpr uint32_t OFF_A = 0;
    static constexpr uint32_t OFF_B = OFF_A + NST * A_STAGE;
    static constexpr uint32_t OFF_OUT = OFF_B + NST * B_STAGE;    // [half][2] chunks on their way out (BM = 64: [2][chunks of a tile])
    static constexpr uint32_t OFF_BAR = OFF_OUT + 4 * CHUNK;
    static constexpr uint32_t TOTAL = OFF_BAR + 512 + 1024;
    static_assert(TOTAL <= 227u * 1024u, "shared memory budget");
    static constexpr int T_FULL = 0, T_EMPTY = NST, T_ACC = 2 * NST, T_ACCFREE = T_ACC + 2, T_COUNT = T_ACCFREE + 2;
    static_assert(8 * T_COUNT + 8 <= 512, "barrier area");
};

struct TgShape { int bm, bn; };

struct TgParams {
    int M, K, m_tiles, n_tiles;
    int w_row0, F;               // first row of this layer in the stacked weights; SwiGLU: hidden width (rows from a gate row to its up row)
    int nq, nk;                  // Q/K/V: widths of Q and of K and V
    const float *ss_in;          // [M][slots] partial sums of squares
    int slots;
    float inv_D, eps;
    uint32_t *status;
};

// BM = 128 or 64 rows per CTA. An accumulator of 2 x 64 rows fills all lanes of either CTA: lanes 0-63 hold its 64 rows for the first half of
// the accumulator's columns, lanes 64-127 for the second, so its CTAs each bring gate and up rows of their own half of the output columns.
template <bool SWIGLU, int BN, int BM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTgThreads, 1)
tile_gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_q,
                 const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, const TgParams p)
{
    using S = TgSmem<BN, BM>;
    constexpr int NST = S::NST;
    constexpr int OUT_N = SWIGLU ? BN / 2 : BN;        // output columns of a tile
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    auto bar = [&](int i) -> uint32_t { return base + S::OFF_BAR + 8u * (uint32_t)i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + S::OFF_BAR + 8 * S::T_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = blockIdx.x >> 1, n_pairs = (int)(gridDim.x >> 1);
    const int total = p.m_tiles * p.n_tiles;
    const int my_tiles = pair < total ? (total - pair + n_pairs - 1) / n_pairs : 0;
    // row tiles fastest: the pairs working at the same time share weight rows in the L2
    auto tile_m0 = [&](int it) -> int { return ((pair + it * n_pairs) % p.m_tiles) * (2 * BM) + (int)rank * BM; };
    auto tile_n0 = [&](int it) -> int { return ((pair + it * n_pairs) / p.m_tiles) * OUT_N; };
    const int nk_steps = (p.K + kTgBK - 1) / kTgBK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(bar(S::T_FULL + s), 1);
            mbar_init(bar(S::T_EMPTY + s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar(S::T_ACC + a), 1);
            mbar_init(bar(S::T_ACCFREE + a), 16);     // one arrival per epilogue warp of either CTA
        }
        *abort_flag = 0u;
        fence_mbar_init();
        prefetch_tmap(&tm_x); prefetch_tmap(&tm_w); prefetch_tmap(&tm_q);
    }
    if (warp == 1) tmem_alloc2(smem_u32((const void *)tmem_slot), 2 * BN);
    tc_fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();   // both CTAs' barriers exist before anything crosses the pair
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    auto load_w = [&](int s, int ks, int n0) {
        // both CTAs' loads complete on the leader's barrier
        if (rank == 0) mbar_expect_tx(bar(S::T_FULL + s), 2 * (S::A_STAGE + S::B_STAGE));
        if constexpr (SWIGLU && BM == 64) {
#pragma unroll
            for (int up = 0; up < 2; ++up)
                tma2_load_2d(base + S::OFF_B + s * S::B_STAGE + up * (S::B_STAGE / 2), &tm_w, bar(S::T_FULL + s) & kPeerBitMask, ks * kTgBK,
                                p.w_row0 + up * p.F + n0 + (int)rank * (BN / 4));
            return;
        }
        const int row = SWIGLU ? p.w_row0 + (int)rank * p.F + n0 : p.w_row0 + n0 + (int)rank * (BN / 2);
        tma2_load_2d(base + S::OFF_B + s * S::B_STAGE, &tm_w, bar(S::T_FULL + s) & kPeerBitMask, ks * kTgBK, row);
    };
    // the weights of the first steps are asked for before the wait for the preceding kernel: nothing in a step writes weights
    const int head = my_tiles > 0 ? (nk_steps < NST ? nk_steps : NST) : 0;
    if (threadIdx.x == 0)
        for (int ks = 0; ks < head; ++ks) load_w(ks, ks, tile_n0(0));
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    auto wait = [&](int i, uint32_t parity, uint32_t code) -> bool {
        if (mbar_try_wait(bar(i), parity)) return true;
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t n = 1;; ++n) {
            if (mbar_try_wait(bar(i), parity)) return true;
            if ((n & 255u) == 0u) {
                if (*abort_flag) return false;
                if (globaltimer_ns() - t_start > kTgWaitNs) break;
            }
        }
        *abort_flag = 1u;
        if (p.status) atomicCAS(p.status, 0u, status_word(kSiteTileGemm + code));
        return false;
    };

    if (warp == 0) {
        // ---------------- TMA producer (both CTAs) ----------------
        if (lane == 0) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 1u;                          // parity of the ring's previous round
            for (int it = 0; it < my_tiles && ok; ++it) {
                const int m0 = tile_m0(it), n0 = tile_n0(it);
                for (int ks = 0; ks < nk_steps; ++ks) {
                    const bool first = it == 0 && ks < head;     // the stage is fresh, its weights are on their way
                    if (it > 0 || ks >= NST) ok = wait(S::T_EMPTY + s, ph, 1);
                    if (!ok) break;
                    if (!first) load_w(s, ks, n0);
                    tma2_load_2d(base + S::OFF_A + s * S::A_STAGE, &tm_x, bar(S::T_FULL + s) & kPeerBitMask, ks * kTgBK, m0);
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA; the warp stays converged, one elected lane issues) ----------------
        if (rank == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(2 * BM, BN, false);
            bool ok = true;
            int s = 0;
            uint32_t ph = 0u;
            for (int it = 0; it < my_tiles && ok; ++it) {
                const int buf = it & 1;
                if (it > 1) ok = wait(S::T_ACCFREE + buf, (uint32_t)((it >> 1) - 1) & 1u, 2);
                for (int ks = 0; ks < nk_steps && ok; ++ks) {
                    ok = wait(S::T_FULL + s, ph, 3);
                    if (!ok) break;
                    tc_fence_after();
                    uint64_t ad = umma_desc_sw128(base + S::OFF_A + s * S::A_STAGE, 16, 1024);
                    uint64_t bd = umma_desc_sw128(base + S::OFF_B + s * S::B_STAGE, 16, 1024);
#pragma unroll
                    for (int kk = 0; kk < kTgBK / 16; ++kk) {
                        umma2_ss_elect(tmem + buf * BN, ad, bd, idesc, (ks > 0 || kk > 0) ? 1u : 0u);
                        umma_desc_advance(ad, 32);
                        umma_desc_advance(bd, 32);
                    }
                    umma2_commit_mc_elect(bar(S::T_EMPTY + s), (uint16_t)3);
                    if (++s == NST) { s = 0; ph ^= 1u; }
                }
                if (ok) umma2_commit_mc_elect(bar(S::T_ACC + buf), (uint16_t)3);   // (not after a wait that ran out: the other CTA knows of it by its own wait alone)
            }
        }
    } else if constexpr (BM == 64) {
        // ---------------- epilogue: thread = one row, a quarter of the tile's output columns ----------------
        const int quarter = warp & 3, half = quarter >> 1, part = (warp - 2) >> 2;
        const int row = (quarter & 1) * 32 + lane;
        constexpr int CW = OUT_N / 2, CPT = CW / 2;                   // output columns of a lane half, of a thread (32 or 16)
        constexpr int CHUNKS = OUT_N / 64;
        const int col0 = half * CW + part * CPT, ch = col0 / 64, p0 = (col0 & 63) / 8;
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + part * CPT;
        const uint32_t leader_free = mapa(bar(S::T_ACCFREE), 0);
        const bool issuer = lane == 0 && part == 0 && (CHUNKS == 2 ? (quarter & 1) == 0 : quarter == 0);
        auto meet = [&] {                                             // the threads that fill a chunk
            if constexpr (CHUNKS == 2) asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
            else asm volatile("bar.sync 1, 256;" ::: "memory");
        };
        bool ok = true;
#pragma unroll 1
        for (int it = 0; it < my_tiles; ++it) {
            const int m0 = tile_m0(it), n0 = tile_n0(it), buf = it & 1;
            float ss = 0.f;
            {
                const int r = m0 + row < p.M ? m0 + row : p.M - 1;
                const float *src = p.ss_in + (size_t)r * p.slots;
                if ((p.slots & 3) == 0) {
                    for (int j = 0; j < p.slots; j += 4) { const float4 v = *reinterpret_cast<const float4 *>(src + j); ss += (v.x + v.y) + (v.z + v.w); }
                } else {
                    for (int j = 0; j < p.slots; ++j) ss += src[j];
                }
            }
            float rs = rsqrtf(ss * p.inv_D + p.eps);
            ok = wait(S::T_ACC + buf, (uint32_t)(it >> 1) & 1u, 4) && ok;
            if (!ok) rs = __int_as_float(0x7fc00000);      // a wait ran out: the tile is marked invalid, not left stale
            tc_fence_after();
            uint32_t acc[CPT];
            if constexpr (CPT == 32) tmem_ld32(taddr + buf * BN, acc);
            else tmem_ld16(taddr + buf * BN, acc);
            if constexpr (SWIGLU) {
                uint32_t up[CPT];
                if constexpr (CPT == 32) tmem_ld32(taddr + buf * BN + CW, up);
                else tmem_ld16(taddr + buf * BN + CW, up);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < CPT; ++i) acc[i] = __float_as_uint(silu_mul(__uint_as_float(acc[i]) * rs, __uint_as_float(up[i]) * rs));
            } else {
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < CPT; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * rs);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(leader_free + 8u * (uint32_t)buf);
            // this tile's staging chunk may still be read by the store issued two tiles ago
            if (issuer) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            if (it > 1) meet();
            const uint32_t stage_off = S::OFF_OUT + (uint32_t)(buf * CHUNKS + ch) * S::CHUNK;
            uint8_t *rowp = smem + stage_off + row * 128;
#pragma unroll
            for (int i = 0; i < CPT / 8; ++i) {
                uint4 o;
                uint32_t *oo = reinterpret_cast<uint32_t *>(&o);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(acc[8 * i + 2 * k]), __uint_as_float(acc[8 * i + 2 * k + 1]));
                    oo[k] = *reinterpret_cast<uint32_t *>(&h);
                }
                *reinterpret_cast<uint4 *>(rowp + (((p0 + i) ^ (row & 7)) << 4)) = o;      // 128-byte swizzle of the TMA box
            }
            fence_proxy_async_smem();
            meet();
            if (issuer) {
                const int n = n0 + ch * 64;
                if (m0 < p.M) {
                    if constexpr (SWIGLU) {
                        if (n < p.F) tma_store_2d(&tm_q, base + stage_off, n, m0);
                    } else {              // (the widths are multiples of 64: a chunk lies in one tensor)
                        if (n < p.nq) tma_store_2d(&tm_q, base + stage_off, n, m0);
                        else if (n < p.nq + p.nk) tma_store_2d(&tm_k, base + stage_off, n - p.nq, m0);
                        else if (n < p.nq + 2 * p.nk) tma_store_2d(&tm_v, base + stage_off, n - p.nq - p.nk, m0);
                    }
                }
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // (the writes are complete when the grid is)
    } else {
        // ---------------- epilogue: thread (row, half); chunks of 64 output columns ----------------
        const int quarter = warp & 3;                 // the TMEM lane quarter this warp may read
        const int half = (warp - 2) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
        const uint32_t leader_free = mapa(bar(S::T_ACCFREE), 0);
        constexpr int CPT = OUT_N / 64 >= 2 ? OUT_N / 128 : 1;        // chunks per half (one chunk in all: the halves take 32 columns each)
        constexpr bool SPLIT = OUT_N == 64;
        const bool issuer = quarter == 0 && lane == 0 && (!SPLIT || half == 0);
        bool ok = true;
        int parity = 0;                               // which of the half's two staging chunks is next
#pragma unroll 1
        for (int it = 0; it < my_tiles; ++it) {
            const int m0 = tile_m0(it), n0 = tile_n0(it), buf = it & 1;
            float ss = 0.f;
            {
                const int r = m0 + row < p.M ? m0 + row : p.M - 1;
                const float *src = p.ss_in + (size_t)r * p.slots;
                if ((p.slots & 3) == 0) {
                    for (int j = 0; j < p.slots; j += 4) { const float4 v = *reinterpret_cast<const float4 *>(src + j); ss += (v.x + v.y) + (v.z + v.w); }
                } else {
                    for (int j = 0; j < p.slots; ++j) ss += src[j];
                }
            }
            float rs = rsqrtf(ss * p.inv_D + p.eps);
            ok = wait(S::T_ACC + buf, (uint32_t)(it >> 1) & 1u, 4) && ok;
            if (!ok) rs = __int_as_float(0x7fc00000);      // a wait ran out: the tile is marked invalid, not left stale
            tc_fence_after();
#pragma unroll
            for (int cc = 0; cc < CPT; ++cc) {
                const int ch = SPLIT ? 0 : half * CPT + cc;
                // this chunk's staging area may still be read by the store issued two chunks ago
                if (issuer) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                if (SPLIT) asm volatile("bar.sync 1, 256;" ::: "memory");
                else asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
                const uint32_t stage_off = S::OFF_OUT + ((SPLIT ? 0 : half * 2) + parity) * S::CHUNK;
                uint8_t *rowp = smem + stage_off + row * 128;
#pragma unroll
                for (int g = 0; g < (SPLIT ? 1 : 2); ++g) {           // 32 columns at a time
                    const int gc = SPLIT ? half : g;                  // which 32 columns of the chunk
                    uint32_t acc[32];
                    tmem_ld32(tmem + lane_addr + buf * BN + ch * 64 + gc * 32, acc);   // warp-wide: every lane takes part, whatever its row
                    if constexpr (SWIGLU) {
                        uint32_t up[32];
                        tmem_ld32(tmem + lane_addr + buf * BN + BN / 2 + ch * 64 + gc * 32, up);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[i] = __float_as_uint(silu_mul(__uint_as_float(acc[i]) * rs, __uint_as_float(up[i]) * rs));
                    } else {
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) acc[i] = __float_as_uint(__uint_as_float(acc[i]) * rs);
                    }
                    if (cc == CPT - 1 && (SPLIT || g == 1)) {
                        // this warp's last read of the accumulator: the tensor pipe may start the tile after next over it
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(leader_free + 8u * (uint32_t)buf);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint4 o;
                        uint32_t *oo = reinterpret_cast<uint32_t *>(&o);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(acc[8 * i + 2 * k]), __uint_as_float(acc[8 * i + 2 * k + 1]));
                            oo[k] = *reinterpret_cast<uint32_t *>(&h);
                        }
                        // 128-byte swizzle of the TMA box: 16-byte piece j of row r sits at j ^ (r % 8)
                        *reinterpret_cast<uint4 *>(rowp + (((gc * 4 + i) ^ (row & 7)) << 4)) = o;
                    }
                }
                fence_proxy_async_smem();
                if (SPLIT) asm volatile("bar.sync 1, 256;" ::: "memory");
                else asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
                if (issuer) {
                    const int n = n0 + ch * 64;
                    if (m0 < p.M) {
                        if constexpr (SWIGLU) {
                            if (n < p.F) tma_store_2d(&tm_q, base + stage_off, n, m0);
                        } else {              // (the widths are multiples of 64: a chunk lies in one tensor)
                            if (n < p.nq) tma_store_2d(&tm_q, base + stage_off, n, m0);
                            else if (n < p.nq + p.nk) tma_store_2d(&tm_k, base + stage_off, n - p.nq, m0);
                            else if (n < p.nq + 2 * p.nk) tma_store_2d(&tm_v, base + stage_off, n - p.nq - p.nk, m0);
                        }
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                parity ^= 1;
            }
        }
        if (issuer) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // (the writes are complete when the grid is)
    }

    tc_fence_before();
    __syncthreads();
    cluster_arrive_relaxed();
    cluster_wait();   // neither CTA retires while its partner can still touch its shared memory or barriers (nothing to release)
    if (warp == 1) tmem_dealloc2(tmem, 2 * BN);
}

template <bool SWIGLU, int BN, int BM>
cudaError_t launch_tg(const CUtensorMap *m, TgParams p, int n_out, cudaStream_t st)
{
    static std::atomic<unsigned long long> attr_set{0};
    cudaError_t e = once_per_device(attr_set, [] {
        return cudaFuncSetAttribute(tile_gemm_kernel<SWIGLU, BN, BM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TgSmem<BN, BM>::TOTAL);
    });
    if (e != cudaSuccess) return e;
    constexpr int OUT_N = SWIGLU ? BN / 2 : BN;
    p.n_tiles = (n_out + OUT_N - 1) / OUT_N;
    const int tiles = p.m_tiles * p.n_tiles;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2u * (unsigned)(tiles < 74 ? tiles : 74));
    cfg.blockDim = dim3(kTgThreads);
    cfg.dynamicSmemBytes = TgSmem<BN, BM>::TOTAL;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, tile_gemm_kernel<SWIGLU, BN, BM>, m[0], m[1], m[2], m[3], m[4], p);
    count_launch();
    return e;
}

}  // namespace

// The tile of a problem: the one whose CTAs take in the least, waves over the 74 SM pairs times the rows of x and W that a CTA loads per step.
static TgShape tg_shape(int M, int cols, bool swiglu)
{
    static const TgShape kShapes[] = {{128, 256}, {128, 128}, {64, 256}, {64, 128}, {64, 64}};
    TgShape best = kShapes[0];
    int best_cost = 0x7fffffff;
    for (const TgShape &t : kShapes) {
        if ((t.bm == 64) && (swiglu ? t.bn == 64 : t.bn == 256)) continue;       // (not built)
        const int tiles = ((M + 2 * t.bm - 1) / (2 * t.bm)) * ((cols + t.bn - 1) / t.bn), cost = (tiles + 73) / 74 * (t.bm + t.bn / 2);
        if (cost < best_cost) { best_cost = cost; best = t; }
    }
    return best;
}

bool tile_proj_supported(int mode, int M, int K, int nq, int nk, int F)
{
    if (M < 1 || K % 8 != 0 || (long long)M * (mode == CG_SWIGLU ? F : nq + 2 * nk) > 0x3FFFFFFF) return false;
    return mode == CG_SWIGLU ? F % 8 == 0 : nq % 64 == 0 && nk % 64 == 0;
}

// CG_QKV or CG_SWIGLU of ChainProj for many rows
cudaError_t launch_tile_proj(const ChainProj &a, cudaStream_t st)
{
    const bool swiglu = a.mode == CG_SWIGLU;
    TgParams p = {};
    p.M = a.B * a.R; p.K = a.K; p.w_row0 = a.w_row0; p.F = a.N; p.nq = a.nq; p.nk = a.nk;
    p.ss_in = a.ss_in; p.slots = a.slots_in; p.inv_D = 1.f / (float)a.D; p.eps = a.eps; p.status = a.status;
    const int cols = swiglu ? 2 * a.N : a.N;
    const TgShape t = tg_shape(p.M, cols, swiglu);
    p.m_tiles = (p.M + 2 * t.bm - 1) / (2 * t.bm);
    CUtensorMap m[5];
    if (!tensor_map_2d_bf16(&m[0], a.x, a.K, p.M, t.bm) || !tensor_map_2d_bf16(&m[1], a.W, a.K, a.w_rows, swiglu && t.bm == 64 ? t.bn / 4 : t.bn / 2)) return cudaErrorInvalidValue;
    if (swiglu) {
        if (!tensor_map_2d_bf16(&m[2], a.h, a.N, p.M, t.bm)) return cudaErrorInvalidValue;
        m[3] = m[4] = m[2];
        if (t.bm == 64) return t.bn == 128 ? launch_tg<true, 128, 64>(m, p, a.N, st) : launch_tg<true, 256, 64>(m, p, a.N, st);
        return t.bn == 128 ? launch_tg<true, 128, 128>(m, p, a.N, st) : launch_tg<true, 256, 128>(m, p, a.N, st);
    }
    if (!tensor_map_2d_bf16(&m[2], a.q, a.nq, p.M, t.bm) || !tensor_map_2d_bf16(&m[3], a.k, a.nk, p.M, t.bm) || !tensor_map_2d_bf16(&m[4], a.v, a.nk, p.M, t.bm))
        return cudaErrorInvalidValue;
    if (t.bm == 64) return t.bn == 64 ? launch_tg<false, 64, 64>(m, p, a.N, st) : launch_tg<false, 128, 64>(m, p, a.N, st);
    return t.bn == 128 ? launch_tg<false, 128, 128>(m, p, a.N, st) : launch_tg<false, 256, 128>(m, p, a.N, st);
}

}  // namespace reflex
