// The head product of the M2 Hyena layer (internal header).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

struct m2_plan;

namespace m2h {

bool covered(const m2_plan* pl, int64_t n, int64_t d, int64_t dh);   // heads of 16, bf16, n <= 1024, a spectrum fft_conv.h can invert
// O[b][h 16 + j][t] = sum_{s < n} k_h[t - s] (X1[b][h 16 ..][t] . X2[b][h 16 ..][s]) V[b][h 16 + j][s];  X1, X2, V, O: [B][d][n];
// kt: fp32 [d / 16][period], the long kernels in the time domain, lag u at u mod period, |u| < n
int32_t heads_fwd(const m2_plan* pl, const void* X1, const void* X2, const void* V, const float* kt, int64_t period, void* O, int64_t B,
                  int64_t d, int64_t n, cudaStream_t stream);

}  // namespace m2h
