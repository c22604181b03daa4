// Short causal convolutions as Toeplitz products (internal header).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

struct m2_plan;

namespace m2t {

constexpr int kMaxN = 256;   // longest row
// bf16 plans whose spectrum buffers carry the kernel in the time domain as well (m2f::spectrum): N = 256 and 512
bool has_time_kernel(const m2_plan* pl);
// device address of that part of a spectrum buffer for H channels: fp32 [H][N], lag u at u mod N
const float* time_kernel(const m2_plan* pl, const void* kf, int64_t H);

struct Rows {
    const void* x;    // [B][H][n]
    const float* kt;  // [H / kf_group][N]
    void* y;          // [B][H][n]; must not be x
};
// y = the first n values of the circular convolution of the zero-padded rows (2 n <= N), up to three sets of rows in one launch
int32_t conv(const m2_plan* pl, const Rows* sets, int count, int64_t B, int64_t H, int64_t n, int kf_group, cudaStream_t stream);

// The same on the fifth-generation tensor cores (toeplitz_umma.cu): 160 < n <= 256 on N = 512, n a multiple of 8; conv calls it where it pays
bool umma_pays(const m2_plan* pl, int count, int64_t B, int64_t H, int64_t n);
int32_t conv_umma(const m2_plan* pl, const Rows* sets, int count, int64_t B, int64_t H, int64_t n, int kf_group, cudaStream_t stream);

// Kernel gradient dk[H][n] (fp32) of rows [B][H][n], N = 512, n = 512 circular or causal n <= 256, a multiple of 16 (toeplitz_grad.cu)
bool grad_covers(const m2_plan* pl, int64_t B, int64_t H, int64_t n, bool causal);
int32_t conv_grad(const m2_plan* pl, const void* x, const void* g, float* dk, int64_t B, int64_t H, int64_t n, bool causal, cudaStream_t stream);

}  // namespace m2t
