// fp32 transform kernels for plans whose length is a power of two, 256 to 16384 (internal header).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

struct m2_plan;

namespace m2f {

bool covered(const m2_plan* pl);            // the plan has the tables (order 2 or 3, N a power of two from 256 to 16384)
const std::vector<float4>* host_table(const m2_plan* pl);   // twiddle factors to place at pl->d_fft; null: a length without kernels
cudaError_t prepare(const m2_plan* pl);
cudaError_t prepare_gradients(const m2_plan* pl);   // (part of prepare)
// log2 N if the plan's spectra are stored in the order of these kernels, 0 if they are in plan order
int spectrum_order(const m2_plan* pl);

// k_f = F_N pad(k) / N, fp32, in the kernels' own order (fft_core.cuh, spec_index); kfu != nullptr (N = 512 only): also in the order of
// the tensor-core kernels, kfu[h][k2 / 2][k1] = (re, re', im, im') of the frequencies k1 + 32 k2, k1 + 32 (k2 + 1); kt != nullptr: k
// itself, zero padded, fp32 [H][N]
cudaError_t spectrum(const m2_plan* pl, const float* k, int64_t H, int64_t n, void* kf, void* kfu, float* kt, cudaStream_t stream);
// back to the time domain: kt[h][t] = scale times the first n values of F^-1 of the sum of `parts` buffers [H][N], fp32 [H][n]; a
// spectrum carries its 1 / N already (scale 1 gives the kernel).  both (2 n <= N): kt is [H][2 n], lag u at u mod 2 n for -n <= u < n, lags
// below zero that are rounding only are zero
cudaError_t time_kernel(const m2_plan* pl, const void* kf, int parts, float scale, int64_t H, int64_t n, bool both, float* kt,
                        cudaStream_t stream);
// y = conv(k[h / kf_group], x[b][h]), x / y [B][H][n] contiguous in the plan dtype
cudaError_t conv(const m2_plan* pl, const void* x, const void* kf, void* y, int64_t B, int64_t H, int64_t n, bool causal, int kf_group,
                 cudaStream_t stream);
// dk[h] = sum_b corr(x[b][h], g[b][h]); cudaErrorInvalidValue for the lengths the kernel does not hold (N > 8192)
cudaError_t wgrad(const m2_plan* pl, const void* x, const void* g, float* dk, int64_t B, int64_t H, int64_t n, bool causal,
                  cudaStream_t stream);

}  // namespace m2f
