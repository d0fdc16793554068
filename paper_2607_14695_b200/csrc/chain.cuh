// Internal interface of the chained expert step (chain_gemm.cu, chain_attn.cu, tile_gemm.cu, linear_tc.cu; put together in reflex_api.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace reflex {

enum { CG_RES = 0, CG_QKV = 1, CG_SWIGLU = 2, CG_OUT = 3 };

// Ranges of memory that later kernels of the step read and nothing in it writes: a launch's CTAs ask shares of them into the L2.
struct ChainPrefetch {
    const void *ptr[3];
    unsigned long long bytes[3];      // multiples of 16; 0 = none
};

#ifdef __CUDACC__
// CTA `cta` of `ctas` asks its share (whole 128-byte lines) of every range; called by one converged warp, a line per lane and
// instruction. (As bulk prefetches the requests went through the SM's TMA unit, and loads queued behind them for microseconds.)
__device__ __forceinline__ void chain_prefetch(const ChainPrefetch &pf, unsigned cta, unsigned ctas, int lane)
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (pf.bytes[i] == 0) continue;
        const unsigned lines = (unsigned)((pf.bytes[i] + 127) >> 7);
        for (unsigned l = cta * 32u + (unsigned)lane; l < lines; l += ctas * 32u)
            asm volatile("prefetch.global.L2 [%0];" ::"l"((const char *)pf.ptr[i] + (size_t)l * 128));
        __syncwarp();
    }
}
#endif

// One projection of the chain: out = epilogue(x [M][K] . W [n][K]^T), bf16 operands, fp32 accumulation.
struct ChainProj {
    int mode;                         // CG_*
    const __nv_bfloat16 *x;           // [M][K]
    const __nv_bfloat16 *W;           // stacked [w_rows][K]
    int w_rows, w_row0;               // rows of the stack, first row of this layer
    int B, R, K, N;                   // N: output features (CG_SWIGLU: hidden features F; W holds [gate F; up F] per layer)
    const __nv_bfloat16 *res;         // CG_RES
    __nv_bfloat16 *h, *xg;            // CG_RES: residual stream and h * gate; CG_SWIGLU: h = output; CG_OUT: h = velocity
    const float *gate;                // CG_RES
    float *ss_out;                    // CG_RES: [M][ceil(N / 32)] sums of squares of 32 columns of h each
    const float *ss_in;               // other modes: partial sums of squares of the normalised rows
    int slots_in, D;                  // their number per row; norm width
    float eps;
    __nv_bfloat16 *q, *k, *v;         // CG_QKV
    int nq, nk;
    float *a;                         // CG_OUT
    float dt;
    uint32_t *status;
    ChainPrefetch pf;
};

// Do the chain's projections take this shape (all CTAs of the launch on the SMs at once)?
bool chain_proj_supported(int mode, int M, int K, int N);
cudaError_t launch_chain_proj(const ChainProj &p, cudaStream_t st);
// The same projections for many rows: CG_QKV and CG_SWIGLU (tile_gemm.cu), CG_RES (linear_half.cu, linear_tc.cu; N a multiple of 256, tile_res_slots
// partial sums of squares per row)
bool tile_proj_supported(int mode, int M, int K, int nq, int nk, int F);
cudaError_t launch_tile_proj(const ChainProj &p, cudaStream_t st);
cudaError_t launch_tile_res(const ChainProj &p, cudaStream_t st);
int tile_res_slots(int M, int K, int N);
// h = bf16(a) W_in^T, xg = h * gate, ss_out [M] (one partial sum per row)
cudaError_t launch_chain_in(const float *a, const __nv_bfloat16 *W_in, const float *gate, __nv_bfloat16 *h, __nv_bfloat16 *xg, float *ss_out, int B,
                            int R, int D, int A, cudaStream_t st);

}  // namespace reflex
