// Short causal convolutions (bf16, n <= 512) as Toeplitz products: y[b][t] = sum_s k[t - s] x[b][s] per channel.
//
// For n this short the n^2 / 2 products per row, done by matrix instructions, cost less than a transform of 2 n points goes through in
// hand-offs and padding: x is read once, y written once, nothing else moves.  M = 16 batch rows, N = 8 positions t, K = 16 positions s;
// a tile of the Toeplitz factor depends on t - s only, so its fragment for distance d (in steps of 8) is one word per lane of a table
// P[u] = (k[u], k[u - 1]), the second half of one fragment is the first half of the next, and a warp that walks s re-reads nothing.
// The kernel is fp32: its values are split into two bf16 parts (16 bits of mantissa) and both are multiplied, so the result differs
// from the exact sum by less than the rounding of the output.  Lags below zero exist when the spectrum was conjugated (the
// transposed convolution); a direction without a non-zero value is not walked.
//
// One block per channel and 32 (16) batch rows, a warp takes tiles of 16 positions from both ends.  Bound by the matrix pipe: 2 x 2 x 136
// instruction pairs of n = 256 per 16 rows, 0.47 instructions per cycle and SM.
// Measured, one B200: the three short convolutions of the Hyena layer at [32][768][256] in one launch, layer 131 -> 115 us.
#include "m2_plan.h"
#include "mma_sync.cuh"
#include "toeplitz_mma.h"

namespace m2t {

constexpr int kThreads = 256;

__host__ __device__ constexpr int padded(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ constexpr int pitch(int n) { return padded(n) + 8; }   // bf16 elements: rows 16 bytes apart mod 128
__host__ __device__ constexpr int smem_bytes(int n, int rows) { return 2 * rows * pitch(n) * 2 + 4 * padded(n) * 4; }

struct Sets {
    Rows r[3];
};

template <int MT>
__global__ void __launch_bounds__(kThreads)
    toeplitz_kernel(const Sets sets, int B, int H, int n, int N, int kf_group) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kRows = 16 * MT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int np = padded(n), ld = pitch(n);
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem);
    __nv_bfloat16* ys = xs + kRows * ld;
    uint32_t* ph = reinterpret_cast<uint32_t*>(ys + kRows * ld);   // P[u] at u + np, upper parts
    uint32_t* pl = ph + 2 * np;                                     // lower parts
    const int h = blockIdx.x % H, b0 = (blockIdx.x / H) * kRows;
    const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(sets.r[blockIdx.y].x);
    __nv_bfloat16* y = static_cast<__nv_bfloat16*>(sets.r[blockIdx.y].y);
    const float* kt = sets.r[blockIdx.y].kt + (size_t)(h / kf_group) * N;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (n % 8 == 0) {   // 16-byte pieces never straddle a row
        const int per_row = np / 8;
        for (int i = tid; i < kRows * per_row; i += kThreads) {
            const int r = i / per_row, c = (i % per_row) * 8, b = b0 + r;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (b < B && c < n) v = __ldg(reinterpret_cast<const uint4*>(x + ((size_t)b * H + h) * n + c));
            *reinterpret_cast<uint4*>(xs + r * ld + c) = v;
        }
    } else {
        for (int i = tid; i < kRows * np; i += kThreads) {
            const int r = i / np, c = i % np, b = b0 + r;
            xs[r * ld + c] = b < B && c < n ? x[((size_t)b * H + h) * n + c] : __float2bfloat16_rn(0.f);
        }
    }
    bool later = false, earlier = false;   // non-zero lags on either side
    for (int i = tid; i < 2 * np; i += kThreads) {
        const int u = i - np;
        const float a = u > -n && u < n ? __ldg(kt + (u & (N - 1))) : 0.f, b = u - 1 > -n && u - 1 < n ? __ldg(kt + ((u - 1) & (N - 1))) : 0.f;
        later = later || (u > 0 && a != 0.f);
        earlier = earlier || (u < 0 && a != 0.f);
        const uint32_t w = bf2(a, b);
        ph[i] = w;
        pl[i] = bf2(a - __uint_as_float(w << 16), b - __uint_as_float(w & 0xffff0000u));
    }
    later = __syncthreads_or(later);
    earlier = __syncthreads_or(earlier);
    const int m8 = lane >> 3, r8 = lane & 7, g = lane >> 2, c2 = 2 * (lane & 3);
    const uint32_t ax = smem_addr(xs + ((m8 & 1) * 8 + r8) * ld + (m8 >> 1) * 8);
    const int tiles = np / 16, nw = kThreads / 32;
    const int front = nw * ((tiles + 2 * nw - 1) / (2 * nw));   // the first half of a warp's tiles in order, the second from the far end:
    for (int it = warp; it < tiles; it += nw) {                 // every warp gets as many short tiles as long ones
        const int ti = it < front ? it : tiles - 1 - (it - front);
        const int s0 = later ? 0 : ti, s1 = earlier ? tiles - 1 : ti;
        float o[MT][2][4] = {};
        const uint32_t* qh = ph + np + g - c2 + 16 * (ti - s0);
        const uint32_t* ql = pl + np + g - c2 + 16 * (ti - s0);
        uint32_t h1 = qh[8], l1 = ql[8];
        for (int si = s0; si <= s1; ++si, qh -= 16, ql -= 16) {
            const uint32_t h0 = qh[0], hm = qh[-8], l0 = ql[0], lm = ql[-8];
            uint32_t fa[MT][4];
#pragma unroll
            for (int m = 0; m < MT; ++m) ldsm4(fa[m], ax + m * 32 * ld + si * 32);
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                mma(o[m][0], fa[m], h0, hm);
                mma(o[m][1], fa[m], h1, h0);
            }
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                mma(o[m][0], fa[m], l0, lm);
                mma(o[m][1], fa[m], l1, l0);
            }
            h1 = hm;
            l1 = lm;
        }
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                __nv_bfloat16* d = ys + (m * 16 + g) * ld + ti * 16 + e * 8 + c2;
                *reinterpret_cast<uint32_t*>(d) = bf2(o[m][e][0], o[m][e][1]);
                *reinterpret_cast<uint32_t*>(d + 8 * ld) = bf2(o[m][e][2], o[m][e][3]);
            }
    }
    __syncthreads();
    if (n % 8 == 0) {
        const int per_row = n / 8;
        for (int i = tid; i < kRows * per_row; i += kThreads) {
            const int r = i / per_row, c = (i % per_row) * 8, b = b0 + r;
            if (b < B) *reinterpret_cast<uint4*>(y + ((size_t)b * H + h) * n + c) = *reinterpret_cast<const uint4*>(ys + r * ld + c);
        }
    } else {
        for (int i = tid; i < kRows * n; i += kThreads) {
            const int r = i / n, c = i % n, b = b0 + r;
            if (b < B) y[((size_t)b * H + h) * n + c] = ys[r * ld + c];
        }
    }
}

bool has_time_kernel(const m2_plan* pl) { return pl->dtype == M2_BF16 && pl->d_fft != nullptr && pl->N >= 256 && pl->N <= 1024; }

const float* time_kernel(const m2_plan* pl, const void* kf, int64_t H) {
    const int64_t orders = pl->N == 512 && pl->umma != nullptr ? 2 : 1;   // (the tensor-core order of the 32 x 16 plan lies in between)
    return reinterpret_cast<const float*>(static_cast<const unsigned char*>(kf) + orders * H * pl->N * 8);
}

int32_t conv(const m2_plan* pl, const Rows* sets, int count, int64_t B, int64_t H, int64_t n, int kf_group, cudaStream_t stream) {
    if (!has_time_kernel(pl) || n > kMaxN || 2 * n > pl->N || count < 1 || count > 3) return M2_ERR_UNSUPPORTED;
    Sets s;
    for (int i = 0; i < 3; ++i) s.r[i] = sets[i < count ? i : 0];
    const int rows = B <= 16 ? 16 : 32;
    const int64_t blocks = H * ((B + rows - 1) / rows);
    if (blocks == 0) return M2_OK;
    if (blocks > 0x7fffffffLL) return M2_ERR_UNSUPPORTED;
    auto kern = rows == 16 ? toeplitz_kernel<1> : toeplitz_kernel<2>;
    const int smem = smem_bytes((int)n, rows);
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(kMaxN, rows)) != cudaSuccess)
        return M2_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks, (unsigned)count);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, s, (int)B, (int)H, (int)n, (int)pl->N, kf_group) != cudaSuccess) return M2_ERR_CUDA;
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2t
