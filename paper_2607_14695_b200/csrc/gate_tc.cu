// Gate MLP of AdaRMSNorm (Eq. 2) on the tensor cores: gamma_l(c) = 1 + W2_l SiLU(W1_l c + b1_l) + b2_l for L layers
// (stacked weights) and B streams, bf16 weights and conditioning vectors.
//
// Both layers of the MLP are the same small GEMM, out[b][u] = act(bias[u] + sum_k W[u][k] vec[b][k]): one CTA takes 128
// weight rows (the M of a tcgen05.mma, K-major A operand) and up to 32 streams (N, K-major B operand), loads both
// operands whole with TMA (80 KB + 20 KB at the paper's widths), issues len/16 MMAs into a 32-column accumulator in
// tensor memory and finishes with one thread per weight row. bf16 x bf16 products are exact in the fp32 accumulator. The
// hidden activations go to the second layer as two bf16 arrays, hi = bf16(h) and lo = bf16(h - hi) (two passes of MMAs,
// about 17 bits of h), in the space the fp32 hidden activations of the FMA kernels take.
//
// Why not CUDA cores: the whole MLP is 0.8 GFLOP per denoising step at 64 streams, but as fp32 FMAs fed from shared
// memory it took 45 us per step (27 us for a single stream); mma.sync runs at a small fraction of tcgen05's rate on
// this part (82 us). Here the cost is the 12 MB of weights and the latency of one load-compute-store round.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "reflex_internal.cuh"
#include "sm100_ptx.cuh"

namespace reflex {

using namespace ptx;

namespace {

constexpr int kGtUnits = 128;     // weight rows per CTA
constexpr int kGtStreams = 32;    // streams per group
constexpr int kGtPerSm = 2;       // CTAs that fit on an SM
constexpr int kGtMaxChunks = 5;   // 64-column chunks of the contraction axis held in shared memory (len <= 320)
constexpr uint32_t kGtWaitNs = 1000000000u;

// Shared memory holds just the chunks that the contraction has, so that two CTAs share an SM (100 KB and 97 KB for the layers of an
// expert): its 37 x 8 second-layer CTAs are one wave instead of two, and they move in beside the first layer's. Both layers of the
// MLP, 37 gates of 1024: 1 stream 11.3 -> 7.6 us, 13 11.9 -> 8.5, 64 14.6 -> 13.3; 4 gates and 64 streams 10.1 -> 7.6 (groups of 32
// instead of 64 streams: twice the CTAs).
struct GateTcSmem {
    static constexpr uint32_t A_CHUNK = kGtUnits * 128;      // 128 rows x 64 bf16
    static constexpr uint32_t B_CHUNK = kGtStreams * 128;    // 32 rows x 64 bf16
    static constexpr uint32_t OFF_BAR = 0;
    static constexpr uint32_t OFF_A = 1024;
    static __host__ __device__ constexpr uint32_t off_b(int chunks) { return OFF_A + chunks * A_CHUNK; }                                  // one or two passes (hi, lo)
    static __host__ __device__ constexpr uint32_t total(int chunks, int passes) { return off_b(chunks) + passes * chunks * B_CHUNK + 1024; }   // + slack for the alignment
};
static_assert(kGtPerSm * (GateTcSmem::total(kGtMaxChunks, 1) + 1024) <= 228 * 1024, "two first-layer CTAs per SM");

// SILU: first layer (writes hi/lo bf16 hidden activations); else second layer (writes fp32 gates 1 + z). PASSES: 1 = one
// bf16 vector per stream (tm_v0), 2 = hi and lo halves (tm_v0, tm_v1).
template <bool SILU, int PASSES>
__global__ void __launch_bounds__(256, kGtPerSm)
gate_tc_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_v0, const __grid_constant__ CUtensorMap tm_v1,
               const __nv_bfloat16 *bias, float *out_f32, __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, int B, int len, int units,
               int vec_rows_per_layer, uint32_t *status)
{
    using S = GateTcSmem;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t *smem = smem_raw + (base - raw_addr);
    const uint32_t bar_load = base + S::OFF_BAR, bar_mma = bar_load + 8;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem + S::OFF_BAR + 16);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int layer = blockIdx.z, u0 = blockIdx.x * kGtUnits;
    const int chunks = (len + 63) / 64;
    const uint32_t off_b = S::off_b(chunks);
    // A CTA keeps its 128 weight rows in shared memory and walks the groups of 32 streams that fall to it (blockIdx.y takes
    // a contiguous share of the groups): with many streams -- the conditioning vectors of all steps of a control tick
    // stacked -- the weights are fetched once per CTA instead of once per group, and the next group's vectors come in
    // while this group's results are stored.
    const int n_groups = (B + kGtStreams - 1) / kGtStreams;
    const int gpc = (n_groups + (int)gridDim.y - 1) / (int)gridDim.y;
    const int g_first = (int)blockIdx.y * gpc;
    const int ng = max(0, min(n_groups, g_first + gpc) - g_first);

    if (threadIdx.x == 0) {
        mbar_init(bar_load, 1);
        mbar_init(bar_mma, 1);
        fence_mbar_init();
        prefetch_tmap(&tm_w); prefetch_tmap(&tm_v0);
        if (PASSES == 2) prefetch_tmap(&tm_v1);
    }
    // weights and (first group of) vectors on one barrier. The second layer asks for its weights before the wait for the first layer's
    // kernel: that kernel writes none, and whatever precedes the call was complete before this one could start.
    auto load_weights = [&]() {
        mbar_expect_tx_elect(bar_load, (uint32_t)chunks * (S::A_CHUNK + PASSES * S::B_CHUNK));
        for (int c = 0; c < chunks; ++c) tma_load_2d_elect(base + S::OFF_A + c * S::A_CHUNK, &tm_w, bar_load, c * 64, layer * units + u0);
    };
    if (warp == 0) {
        __syncwarp();
        if (!SILU && ng > 0) load_weights();
    }
    if (warp == 1) tmem_alloc(smem_u32((const void *)tmem_slot), kGtStreams);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    // programmatic dependent launch: the first layer's output (second kernel) or whatever precedes the call is complete
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    auto wait = [&](uint32_t bar, uint32_t parity, uint32_t code) -> bool {
        if (mbar_try_wait(bar, parity)) return true;
        const unsigned long long t_start = globaltimer_ns();
        for (uint32_t n = 1;; ++n) {
            if (mbar_try_wait(bar, parity)) return true;
            if ((n & 255u) == 0u && globaltimer_ns() - t_start > kGtWaitNs) break;
        }
        if (status) atomicCAS(status, 0u, status_word(kSiteGate + code));
        return false;
    };
    auto load_vectors = [&](int g) {   // the (up to) 32 vectors of group g, one or two bf16 arrays (the warp is converged)
        for (int c = 0; c < chunks; ++c) {
            tma_load_2d_elect(base + off_b + c * S::B_CHUNK, &tm_v0, bar_load, c * 64, layer * vec_rows_per_layer + g * kGtStreams);
            if (PASSES == 2)
                tma_load_2d_elect(base + off_b + (chunks + c) * S::B_CHUNK, &tm_v1, bar_load, c * 64, layer * vec_rows_per_layer + g * kGtStreams);
        }
    };

    bool ok = true;
    if (warp == 0 && ng > 0) {
        if (SILU) load_weights();
        load_vectors(g_first);
    }
    const int quarter = warp & 3, half = warp >> 2;
    const int u = u0 + quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const float bi = u < units ? __bfloat162float(bias[(size_t)layer * units + u]) : 0.f;
#pragma unroll 1
    for (int i = 0; i < ng; ++i) {
        const int b0 = (g_first + i) * kGtStreams;
        const uint32_t ph = (uint32_t)i & 1u;
        if (warp == 0) {
            // the whole warp stays converged; one elected lane issues
            ok = ok && wait(bar_load, ph, 1);
            tc_fence_after();
            if (ok) {
                constexpr uint32_t idesc = umma_idesc_bf16(kGtUnits, kGtStreams, false);
#pragma unroll 1
                for (int pass = 0; pass < PASSES; ++pass) {
#pragma unroll 1
                    for (int c = 0; c < chunks; ++c) {      // (columns past the contraction's end are zeros on both sides)
                        uint64_t ad = umma_desc_sw128(base + S::OFF_A + c * S::A_CHUNK, 16, 1024);
                        uint64_t bd = umma_desc_sw128(base + off_b + (pass * chunks + c) * S::B_CHUNK, 16, 1024);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            umma_ss_elect(tmem, ad, bd, idesc, (pass > 0 || c > 0 || kk > 0) ? 1u : 0u);
                            umma_desc_advance(ad, 32);
                            umma_desc_advance(bd, 32);
                        }
                    }
                }
            }
            if (ok) umma_commit_elect(bar_mma);   // (when the load never came, the other warps learn of it by their own wait)
        }
        ok = wait(bar_mma, ph, 2) && ok;
        tc_fence_after();
        // the MMAs that read this group's vectors are complete: the next group's may land on them
        if (warp == 0 && i + 1 < ng) {
            mbar_expect_tx_elect(bar_load, (uint32_t)chunks * (PASSES * S::B_CHUNK));
            load_vectors(g_first + i + 1);
        }
        // epilogue: thread = weight row (TMEM lane), columns = streams, the two warps of a lane quarter take half each in groups of eight.
        // Groups without a stream are skipped by a branch: as predicated code over all 64 columns the SiLU layer's epilogue took 4.7 us
        // for a single stream.
        const int nb = min(kGtStreams, B - b0);
#pragma unroll 1
        for (int g = 0; g < kGtStreams / 16; ++g) {
            const int n0 = half * (kGtStreams / 2) + g * 8;
            if (n0 >= nb) break;
            uint32_t acc[8];
            tmem_ld8(tmem + lane_addr + n0, acc);
            tmem_wait_ld();
            if (u < units) {
                const size_t o0 = ((size_t)layer * B + b0 + n0) * units + u;
#pragma unroll
                for (int n = 0; n < 8; ++n) {
                    // (after a bounded wait that ran out this CTA's slice of the output is marked invalid, a quiet NaN, instead of keeping
                    // the previous call's values: whatever consumes the gates shows it)
                    const float z = ok ? __uint_as_float(acc[n]) + bi : __int_as_float(0x7fc00000);
                    if (n0 + n >= nb) continue;
                    if (SILU) {
                        const float h = z / (1.f + expf(-z));
                        const __nv_bfloat16 hi = __float2bfloat16_rn(h);
                        out_hi[o0 + (size_t)n * units] = hi;
                        out_lo[o0 + (size_t)n * units] = __float2bfloat16_rn(h - __bfloat162float(hi));
                    } else {
                        out_f32[o0 + (size_t)n * units] = 1.f + z;
                    }
                }
            }
        }
        tc_fence_before();
        __syncthreads();      // every warp has read its accumulators: the next group's MMAs may overwrite them
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kGtStreams);
}

template <bool SILU, int PASSES>
cudaError_t launch_one(const CUtensorMap &mw, const CUtensorMap &mv0, const CUtensorMap &mv1, const __nv_bfloat16 *bias, float *out_f32,
                       __nv_bfloat16 *out_hi, __nv_bfloat16 *out_lo, int L, int B, int len, int units, int vec_rows_per_layer, cudaStream_t st)
{
    static std::atomic<unsigned long long> attr_set{0};
    cudaError_t e0 = once_per_device(attr_set, [] {
        return cudaFuncSetAttribute(gate_tc_kernel<SILU, PASSES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GateTcSmem::total(kGtMaxChunks, PASSES));
    });
    if (e0 != cudaSuccess) return e0;
    cudaLaunchConfig_t cfg = {};
    // groups of 32 streams are spread over blockIdx.y only as far as that adds CTAs the SMs can hold at once; beyond, a CTA
    // walks several groups with its weights resident
    const int ux = (units + kGtUnits - 1) / kGtUnits, n_groups = (B + kGtStreams - 1) / kGtStreams;
    int gy = 148 * kGtPerSm / (ux * L);
    gy = gy < 1 ? 1 : (gy > n_groups ? n_groups : gy);
    cfg.gridDim = dim3(ux, gy, L);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = GateTcSmem::total((len + 63) / 64, PASSES);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, gate_tc_kernel<SILU, PASSES>, mw, mv0, mv1, bias, out_f32, out_hi, out_lo, B, len, units,
                                       vec_rows_per_layer, (uint32_t *)nullptr);
    count_launch();
    return e;
}

}  // namespace

bool gate_tc_supported(int B, int D, int Cd, int Hd)
{
    if (B < 1 || Cd % 16 != 0 || Hd % 16 != 0 || Cd > 64 * kGtMaxChunks || Hd > 64 * kGtMaxChunks) return false;
    return D % 8 == 0;
}

cudaError_t launch_gate_tc(const void *cond, const void *W1, const void *b1, const void *W2, const void *b2, float *gate_buf, int L, int B,
                           int D, int Cd, int Hd, cudaStream_t st)
{
    // scratch behind the gates: hi and lo halves of the hidden activations, [L][B][Hd] bf16 each (the space of [L][B][Hd] floats)
    __nv_bfloat16 *hid_hi = reinterpret_cast<__nv_bfloat16 *>(gate_buf + (size_t)L * B * D);
    __nv_bfloat16 *hid_lo = hid_hi + (size_t)L * B * Hd;
    CUtensorMap mw1, mw2, mc, mhi, mlo;
    if (!tensor_map_2d_bf16(&mw1, W1, Cd, L * Hd, kGtUnits) || !tensor_map_2d_bf16(&mw2, W2, Hd, L * D, kGtUnits) ||
        !tensor_map_2d_bf16(&mc, cond, Cd, B, kGtStreams) || !tensor_map_2d_bf16(&mhi, hid_hi, Hd, L * B, kGtStreams) ||
        !tensor_map_2d_bf16(&mlo, hid_lo, Hd, L * B, kGtStreams))
        return cudaErrorInvalidValue;
    cudaError_t e = launch_one<true, 1>(mw1, mc, mc, (const __nv_bfloat16 *)b1, nullptr, hid_hi, hid_lo, L, B, Cd, Hd, 0, st);
    if (e != cudaSuccess) return e;
    return launch_one<false, 2>(mw2, mhi, mlo, (const __nv_bfloat16 *)b2, gate_buf, nullptr, nullptr, L, B, Hd, D, B, st);
}

}  // namespace reflex
