// The residual projections of a few hundred rows: out = res + a W^T as pair tiles of 128 rows, the contraction in two halves.
//
// What bounds these shapes is what the SMs at work take in from the L2, 50 to 58 bytes per cycle each. Tiles of 256 rows leave half of the SMs
// idle: 429 rows x 1024 columns are 16 tiles of 256 x 128, which with the contraction halved are 64 CTAs, each taking in
// 786 KB of a 4096-long contraction. Here a CTA of a pair (cta_group::2, M = 128) owns 64 rows, so that the same problem is 128 CTAs with 524 KB
// each; a cluster is the two pairs that share a tile's contraction. 64-column tiles while those still are at most 32 clusters (up to 256
// rows of 1024 columns), 128-column tiles above.
// Measured against the tiles of 256 rows, contraction split the same way (graph replay, in place, 1024 columns): 264 rows x 2048 7.9 -> 6.2 us, x 4096
// 11.2 -> 9.3; 429 rows 7.9 -> 6.5 and 11.3 -> 9.8; 512 rows 7.9 -> 6.5 and 11.4 -> 9.9. Narrow outputs of more rows in as many tiles are served alike: 4000
// rows x 4096 -> 64 columns 10.8 -> 8.9, 2000 x 4096 -> 256 11.0 -> 9.2; of 45 shapes of 512 to 4000 rows x 2048 to 12288 -> 32 to 1024 none is slower.
//
// An accumulator of 128 rows over a pair fills all lanes of either CTA: lanes 0-63 hold its 64 rows for the first half of the columns, lanes
// 64-127 for the second. The halves of the contraction meet by rows: either CTA of the two with equal rank finishes 32 of their 64 rows, the
// warps of its other rows send theirs straight from tensor memory (st.async, counted on the receiver's barrier, 512 contiguous bytes a warp).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "chain.cuh"
#include "linear_half.cuh"
#include "reflex_internal.cuh"
#include "sm100_ptx.cuh"

namespace reflex {

using namespace ptx;

namespace {

constexpr int kLhThreads = 64 + 256;      // producer warp, MMA warp, eight epilogue warps
constexpr int kLhRows = 64;               // rows per CTA (128 per pair)
constexpr int kLhOwn = 32;                // rows a CTA finishes
constexpr int kLhMinR = 4;                // rows per stream at least, where gates are asked for
constexpr unsigned long long kLhWaitNs = 1000000000ull;

template <int BN>
struct LhSmem {
    static constexpr int NST = BN == 128 ? 10 : 13;
    static constexpr uint32_t A_STAGE = kLhRows * 128;
    static constexpr uint32_t B_STAGE = (BN / 2) * 128;
    static constexpr uint32_t CHUNK = kLhOwn * 128;                          // 32 rows x 64 columns of the residual / output tile
    static constexpr uint32_t OFF_A = 0;
    static constexpr uint32_t OFF_B = OFF_A + NST * A_STAGE;
    static constexpr uint32_t OFF_RES = OFF_B + NST * B_STAGE;               // residual in, output out
    static constexpr uint32_t OFF_XG = OFF_RES + (BN / 64) * CHUNK;
    static constexpr uint32_t OFF_IN = OFF_XG + (BN / 64) * CHUNK;           // the counterpart's sums: [column quad][32 rows][4] fp32
    static constexpr uint32_t IN_BYTES = kLhOwn * BN * 4;
    static constexpr uint32_t OFF_GATE = OFF_IN + IN_BYTES;                  // gates of the streams under the rows this CTA finishes
    static constexpr uint32_t GATE_BYTES = (kLhOwn / kLhMinR + 1) * BN * 4;
    static constexpr uint32_t OFF_SS = OFF_GATE + GATE_BYTES;                // [4][32] sums of squares
    static constexpr uint32_t OFF_BAR = OFF_SS + 4 * kLhOwn * 4;
    static constexpr uint32_t TOTAL = OFF_BAR + 256 + 1024;
    static constexpr int C_FULL = 0, C_EMPTY = NST, C_ACC = 2 * NST, C_RES = C_ACC + 1, C_IN = C_ACC + 2, C_COUNT = C_ACC + 3;
    static_assert(TOTAL <= 227u * 1024u && 8 * C_COUNT + 8 <= 256, "shared memory budget");
};

struct LhParams {
    const float *gate;    // [B][N], or NULL: neither out * gate nor sums of squares are written
    float *ss_out;        // [M][n_tiles]
    int R, B;
    int M, K, N;
    int m_tiles, n_tiles;
    int has_res, early_w;
    uint32_t *status;
};

template <int BN>
__global__ void __cluster_dims__(4, 1, 1) __launch_bounds__(kLhThreads, 1)
linear_half_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_res,
                   const __grid_constant__ CUtensorMap tm_out, const __grid_constant__ CUtensorMap tm_xg, const LhParams p)
{
    using S = LhSmem<BN>;
    constexpr int NST = S::NST;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    auto bar = [&](int i) -> uint32_t { return base + S::OFF_BAR + 8u * (uint32_t)i; };
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + S::OFF_BAR + 8 * S::C_COUNT);
    volatile uint32_t *abort_flag = tmem_slot + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t crank = cluster_ctarank();
    const uint32_t rank = crank & 1u;                             // rank inside the pair
    const int kq = (int)(crank >> 1);                             // which half of the contraction this pair takes, and of its rows a CTA finishes
    const uint16_t pair_mask = (uint16_t)(3u << (crank & ~1u));
    const int tile = blockIdx.x >> 2;
    const int m0 = (tile % p.m_tiles) * (2 * kLhRows) + (int)rank * kLhRows;
    const int mo = m0 + kq * kLhOwn;                              // first row this CTA finishes
    const int n0 = (tile / p.m_tiles) * BN;
    const int steps = ((p.K + 63) / 64) / 2, k_first = kq * steps;

    if (threadIdx.x == 0) {
        for (int i = 0; i < S::C_COUNT; ++i) mbar_init(bar(i), 1);
        *abort_flag = 0u;
        fence_mbar_init();
        mbar_expect_tx(bar(S::C_IN), S::IN_BYTES);
        prefetch_tmap(&tm_a); prefetch_tmap(&tm_w); prefetch_tmap(&tm_out);
        if (p.has_res) prefetch_tmap(&tm_res);
    }
    if (warp == 1) tmem_alloc2(smem_u32((const void *)tmem_slot), BN);
    tc_fence_before();
    __syncthreads();
    cluster_arrive();
    cluster_wait();   // all barriers of the cluster exist before anything crosses it
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    auto load_w = [&](int s, int ks) {
        // both CTAs' loads complete on the leader's barrier
        if (rank == 0) mbar_expect_tx(bar(S::C_FULL + s), 2 * (S::A_STAGE + S::B_STAGE));
        tma2_load_2d(base + S::OFF_B + s * S::B_STAGE, &tm_w, bar(S::C_FULL + s) & kPeerBitMask, (k_first + ks) * 64, n0 + (int)rank * (BN / 2));
    };
    // inside an expert step the weights of the first steps are asked for ahead of the wait for the preceding kernel
    const int head = p.early_w ? min(steps, NST) : 0;
    if (threadIdx.x == 0)
        for (int ks = 0; ks < head; ++ks) load_w(ks, ks);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    auto wait_slow = [&](int i, uint32_t parity, uint32_t code) -> bool {
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t n = 1;; ++n) {
            if (mbar_try_wait_cluster(bar(i), parity)) return true;
            if ((n & 255u) == 0u) {
                if (*abort_flag) return false;
                if (globaltimer_ns() - t_start > kLhWaitNs) break;
            }
        }
        *abort_flag = 1u;
        if (p.status) atomicCAS(p.status, 0u, status_word(kSiteLinearHalf + code));
        return false;
    };
    auto wait = [&](int i, uint32_t parity, uint32_t code) -> bool { return mbar_try_wait(bar(i), parity) || wait_slow(i, parity, code); };

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            bool ok = true;
            int s = 0;
            uint32_t ph = 1u;                          // parity of the ring's previous round
            for (int ks = 0; ks < steps; ++ks) {
                if (ks >= NST) ok = wait(S::C_EMPTY + s, ph, 1);
                if (!ok) break;
                if (ks >= head) load_w(s, ks);
                tma2_load_2d(base + S::OFF_A + s * S::A_STAGE, &tm_a, bar(S::C_FULL + s) & kPeerBitMask, (k_first + ks) * 64, m0);
                if (++s == NST) { s = 0; ph ^= 1u; }
            }
            if (p.has_res) {
                mbar_expect_tx(bar(S::C_RES), (BN / 64) * S::CHUNK);
#pragma unroll
                for (int c = 0; c < BN / 64; ++c) tma_load_2d(base + S::OFF_RES + c * S::CHUNK, &tm_res, bar(S::C_RES), n0 + c * 64, mo);
            } else {
                mbar_arrive(bar(S::C_RES));
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA; the warp stays converged, one elected lane issues) ----------------
        if (rank == 0) {
            constexpr uint32_t idesc = umma_idesc_bf16(2 * kLhRows, BN, false);
            bool ok = true;
            int s = 0;
            uint32_t ph = 0u;
            for (int ks = 0; ks < steps; ++ks) {
                ok = wait(S::C_FULL + s, ph, 2);
                if (!ok) break;
                tc_fence_after();
                uint64_t ad = umma_desc_sw128(base + S::OFF_A + s * S::A_STAGE, 16, 1024);
                uint64_t bd = umma_desc_sw128(base + S::OFF_B + s * S::B_STAGE, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    umma2_ss_elect(tmem, ad, bd, idesc, (ks > 0 || kk > 0) ? 1u : 0u);
                    umma_desc_advance(ad, 32);
                    umma_desc_advance(bd, 32);
                }
                umma2_commit_mc_elect(bar(S::C_EMPTY + s), pair_mask);
                if (++s == NST) { s = 0; ph ^= 1u; }
            }
            if (ok) umma2_commit_mc_elect(bar(S::C_ACC), pair_mask);   // (not after a wait that ran out: the other CTA knows of it by its own wait alone)
        }
    } else {
        // ---------------- epilogue: thread = one row, a quarter of the columns ----------------
        const int quarter = warp & 3, part = (warp - 2) >> 2;
        const bool mine = (quarter & 1) == kq;                     // this warp's rows are finished here
        constexpr int CPT = BN / 4;                                // columns per thread: 32 or 16
        const int col0 = (quarter >> 1) * (BN / 2) + part * CPT;   // first of them in the tile
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + part * CPT;
        const int b_first = p.gate ? min(mo / p.R, p.B - 1) : 0;
        float *gsm = reinterpret_cast<float *>(smem + S::OFF_GATE);
        if (p.gate) {
            const int n = (min((mo + kLhOwn - 1) / p.R, p.B - 1) - b_first + 1) * (BN / 4);
            for (int i = threadIdx.x - 64; i < n; i += 256)
                reinterpret_cast<float4 *>(gsm)[i] = *reinterpret_cast<const float4 *>(p.gate + (size_t)(b_first + i / (BN / 4)) * p.N + n0 + (i % (BN / 4)) * 4);
            asm volatile("bar.sync 1, 256;" ::: "memory");
        }
        bool ok = wait(S::C_ACC, 0u, 3);
        if (*abort_flag) ok = false;
        tc_fence_after();
        uint32_t acc[CPT];
        if constexpr (CPT == 32) tmem_ld32(taddr, acc);
        else tmem_ld16(taddr, acc);
        tmem_wait_ld();
        if (!mine) {
            if (!ok) {
#pragma unroll
                for (int i = 0; i < CPT; ++i) acc[i] = 0x7fc00000u;
            }
            const uint32_t dst = mapa(base + S::OFF_IN + (uint32_t)((col0 / 4) * kLhOwn + lane) * 16u, crank ^ 2u), ib = mapa(bar(S::C_IN), crank ^ 2u);
#pragma unroll
            for (int i = 0; i < CPT / 4; ++i) st_async_v4(dst + i * (kLhOwn * 16), ib, acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
        } else {
            uint8_t *rowp = smem + S::OFF_RES + (col0 / 64) * S::CHUNK + lane * 128, *xrowp = smem + S::OFF_XG + (col0 / 64) * S::CHUNK + lane * 128;
            const int p0 = (col0 & 63) / 8;                        // first 16-byte piece of the chunk's row; pieces are swizzled: j at j ^ (row % 8)
            ok = wait(S::C_RES, 0u, 4) && ok;
            uint4 rr[CPT / 8];
#pragma unroll
            for (int j = 0; j < CPT / 8; ++j) {
                rr[j] = make_uint4(0u, 0u, 0u, 0u);
                if (p.has_res) rr[j] = *reinterpret_cast<const uint4 *>(rowp + (((p0 + j) ^ (lane & 7)) << 4));
            }
            const float *grow = gsm + (size_t)(p.gate ? min((mo + lane) / p.R, p.B - 1) - b_first : 0) * BN + col0;
            ok = (mbar_try_wait_cluster(bar(S::C_IN), 0u) || wait_slow(S::C_IN, 0u, 5)) && ok;
            const float4 *in = reinterpret_cast<const float4 *>(smem + S::OFF_IN) + (col0 / 4) * kLhOwn + lane;
            float ss = 0.f;
#pragma unroll
            for (int j = 0; j < CPT / 8; ++j) {
                const float4 q0 = in[(2 * j) * kLhOwn], q1 = in[(2 * j + 1) * kLhOwn];
                const float pp[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
                const uint32_t rv[4] = {rr[j].x, rr[j].y, rr[j].z, rr[j].w};
                uint32_t ov[4], xv[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float v0 = __uint_as_float(acc[8 * j + 2 * k]) + pp[2 * k] + __uint_as_float(rv[k] << 16);
                    float v1 = __uint_as_float(acc[8 * j + 2 * k + 1]) + pp[2 * k + 1] + __uint_as_float(rv[k] & 0xFFFF0000u);
                    if (!ok) v0 = v1 = __int_as_float(0x7fc00000);      // a wait ran out: the tile is marked invalid, not left stale
                    __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
                    ov[k] = *reinterpret_cast<uint32_t *>(&h);
                    if (p.gate) {                                       // (the norm takes the sum before its rounding)
                        const float2 g = *reinterpret_cast<const float2 *>(grow + 8 * j + 2 * k);
                        __nv_bfloat162 x = __floats2bfloat162_rn(v0 * g.x, v1 * g.y);
                        xv[k] = *reinterpret_cast<uint32_t *>(&x);
                        ss = fmaf(v0, v0, fmaf(v1, v1, ss));
                    }
                }
                *reinterpret_cast<uint4 *>(rowp + (((p0 + j) ^ (lane & 7)) << 4)) = make_uint4(ov[0], ov[1], ov[2], ov[3]);
                if (p.gate) *reinterpret_cast<uint4 *>(xrowp + (((p0 + j) ^ (lane & 7)) << 4)) = make_uint4(xv[0], xv[1], xv[2], xv[3]);
            }
            float *ssm = reinterpret_cast<float *>(smem + S::OFF_SS);
            ssm[((quarter >> 1) * 2 + part) * kLhOwn + lane] = ss;
            fence_proxy_async_smem();
            asm volatile("bar.sync 2, 128;" ::: "memory");              // the four warps of the finished rows
            if (quarter < 2 && part == 0) {
                if (lane == 0 && mo < p.M) {
#pragma unroll
                    for (int c = 0; c < BN / 64; ++c) {
                        if (n0 + c * 64 < p.N) {
                            tma_store_2d(&tm_out, base + S::OFF_RES + c * S::CHUNK, n0 + c * 64, mo);
                            if (p.gate) tma_store_2d(&tm_xg, base + S::OFF_XG + c * S::CHUNK, n0 + c * 64, mo);
                        }
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                if (p.gate && mo + lane < p.M)
                    p.ss_out[(size_t)(mo + lane) * p.n_tiles + n0 / BN] = (ssm[lane] + ssm[kLhOwn + lane]) + (ssm[2 * kLhOwn + lane] + ssm[3 * kLhOwn + lane]);
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_arrive_relaxed();
    cluster_wait();   // no CTA retires while another can still touch its shared memory or barriers (nothing to release)
    if (warp == 1) tmem_dealloc2(tmem, BN);
}

template <int BN>
cudaError_t lh_launch(const CUtensorMap *m, const LhParams &p, cudaStream_t st)
{
    static std::atomic<unsigned long long> attr_set{0};
    cudaError_t e = once_per_device(attr_set, [] { return cudaFuncSetAttribute(linear_half_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LhSmem<BN>::TOTAL); });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(4u * (unsigned)p.m_tiles * (unsigned)p.n_tiles);
    cfg.blockDim = dim3(kLhThreads);
    cfg.dynamicSmemBytes = LhSmem<BN>::TOTAL;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, linear_half_kernel<BN>, m[0], m[1], m[2], m[3], m[4], p);
    count_launch();
    return e;
}

}  // namespace

// Columns of a tile, or 0: the other kernels take the problem. All clusters of four have to be resident at once (the device holds 33); the exchange
// between the halves pays for itself from a contraction of 2048 on, as in the tiles of 256 rows.
int linear_half_columns(int M, int K, int N)
{
    const int chunks = (K + 63) / 64, m_tiles = (M + 127) / 128;
    if (M <= 64 || chunks % 2 != 0 || chunks < 32) return 0;
    for (int bn = 64; bn <= 128; bn *= 2)
        if (m_tiles * ((N + bn - 1) / bn) <= 32) return bn;
    return 0;
}

int linear_half_slots(int M, int K, int N)
{
    const int bn = linear_half_columns(M, K, N);
    return bn ? (N + bn - 1) / bn : 0;
}

cudaError_t launch_linear_half(const LinearHalf &a, cudaStream_t st)
{
    const int bn = linear_half_columns(a.M, a.K, a.N);
    if (bn == 0 || (a.gate && a.R < kLhMinR)) return cudaErrorInvalidValue;
    LhParams p = {};
    p.gate = a.gate; p.ss_out = a.ss_out; p.R = a.R; p.B = a.B; p.M = a.M; p.K = a.K; p.N = a.N; p.m_tiles = (a.M + 127) / 128; p.n_tiles = (a.N + bn - 1) / bn;
    p.has_res = a.res ? 1 : 0; p.early_w = a.early_w ? 1 : 0; p.status = a.status;
    CUtensorMap m[5];
    if (!tensor_map_2d_bf16(&m[0], a.a, a.K, a.M, kLhRows) || !tensor_map_2d_bf16(&m[1], a.W, a.K, a.N, bn / 2) ||
        !tensor_map_2d_bf16(&m[2], a.res ? a.res : a.out, a.N, a.M, kLhOwn) || !tensor_map_2d_bf16(&m[3], a.out, a.N, a.M, kLhOwn) ||
        !tensor_map_2d_bf16(&m[4], a.xg ? a.xg : a.out, a.N, a.M, kLhOwn))
        return cudaErrorInvalidValue;
    return bn == 64 ? lh_launch<64>(m, p, st) : lh_launch<128>(m, p, st);
}

}  // namespace reflex
