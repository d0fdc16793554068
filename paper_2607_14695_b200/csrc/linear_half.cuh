// Internal interface of linear_half.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace reflex {

struct LinearHalf {
    const void *a, *W, *res;          // [M][K], [N][K], [M][N] or NULL; bf16
    void *out, *xg;                   // [M][N]; xg = out * gate (with gate)
    const float *gate;                // [B][N] of the norm that follows, or NULL
    float *ss_out;                    // with gate: [M][linear_half_slots] sums of squares of the rows
    int M, K, N, R, B;                // R rows per stream (at least 4, with gate)
    bool early_w;                     // weights may be read ahead of the preceding kernel's end
    uint32_t *status;
};

int linear_half_columns(int M, int K, int N);      // columns of a tile; 0: not for this kernel
int linear_half_slots(int M, int K, int N);
cudaError_t launch_linear_half(const LinearHalf &a, cudaStream_t st);

}  // namespace reflex
