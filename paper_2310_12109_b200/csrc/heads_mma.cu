// Head product of the M2 Hyena layer: per (batch entry, head of 16 channels)
//   O[t][j] = sum_i X1[t][i] ( sum_{s <= t} k[t - s] X2[s][i] V[s][j] ) = sum_{s <= t} k[t - s] (X1[t] . X2[s]) V[s][j],
// the causal convolution of the 256 sequences of the outer product X2 V^T with the head's kernel, contracted with X1 (App. "GPT Causal
// Language Modeling").  In the second form the convolution is an n x n Toeplitz factor on the rank-16 scores: two contractions
// with K = 16 and one product per (t, s), against 256 convolutions of 2 n points.
//
// One thread block per (batch entry, head); a warp owns tiles of 16 positions t, one or two neighbouring ones at a time, and walks the tiles
// of 16 positions s <= t.  A tile pair is four m16n8k16 MMAs on register fragments: the scores' accumulator, times the kernel values and rounded to bf16, IS the second
// product's B operand (rows of an accumulator fragment = columns of a B fragment), so nothing goes through shared memory between the
// two products and no warp waits for another.  (tcgen05 would put every tile through tensor memory, shared memory and two barriers for
// 8 K multiply-adds.)  Kernel values lie reversed in shared memory, in two copies one element apart, so that the two values of a
// fragment's column pair are one aligned 64-bit load for even and odd rows alike.  Lags below zero exist where the spectrum was
// conjugated or its kernel is longer than N - n: a block that finds one that is not zero walks the tiles s > t too, with kernel values
// from L2.
//
// Measured, one B200, 1536 heads of n = 256: 23.6 us with one tile at a time, where 24 576 tensor-core convolution units of 16 rows took about
// 280 us, and 22.4 us with two.  Two share the fragments of X2 and V, and a distance's kernel values serve the next one: 6 wavefronts a tile pair instead
// of 14, load/store data pipe 60 -> 40 % busy, issue 48 -> 38 %, for 5 % of the time.  Bound by the latency of a tile pair's chain (fragments, scores,
// weights, second product) with 37 and now 21 warps per SM; matrix pipe 31 -> 34 % of active cycles.
#include "fft_conv.h"
#include "fft_core.cuh"
#include "heads_mma.h"
#include "m2_plan.h"
#include "mma_sync.cuh"

#include <type_traits>

namespace m2h {

constexpr int kDh = 16, kMaxN = 1024;

__host__ __device__ constexpr int padded(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ constexpr int pitch(int n) { return padded(n) + 8; }              // bf16 elements: rows 16 bytes apart mod 128
__host__ __device__ constexpr int kcopy(int n) { return (padded(n) + 31) / 32 * 32 + 48; }   // floats of one reversed copy; copies 16 banks apart
__host__ __device__ constexpr int smem_bytes(int n) { return 3 * kDh * pitch(n) * 2 + 2 * kcopy(n) * 4; }

using m2t::bf2;
using m2t::ldsm4;
using m2t::ldsm4t;
using m2t::mma;
using m2t::smem_addr;

// bf16 pair of the products (a, b) * (k.x, k.y)
__device__ __forceinline__ uint32_t weigh(float a, float b, float2 k) {
    const m2f::u64 p = m2f::mul2(m2f::pk(a, b), m2f::pk(k.x, k.y));
    return bf2(m2f::lo(p), m2f::hi(p));
}

template <int kThreads, int T>   // T: tiles of 16 positions t that a warp takes at a time
__global__ void __launch_bounds__(kThreads, T == 1 ? 5 : 0)   // (T = 1: five blocks per SM, 48 registers without spills)
    heads_kernel(const __nv_bfloat16* __restrict__ X1, const __nv_bfloat16* __restrict__ X2, const __nv_bfloat16* __restrict__ V,
                 const float* __restrict__ kt, int period, __nv_bfloat16* __restrict__ O, int heads, int n) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int np = padded(n), ld = pitch(n), kc = kcopy(n);
    __nv_bfloat16* xs1 = reinterpret_cast<__nv_bfloat16*>(smem);
    __nv_bfloat16* xs2 = xs1 + kDh * ld;
    __nv_bfloat16* vs = xs2 + kDh * ld;
    float* ks = reinterpret_cast<float*>(vs + kDh * ld);
    const int h = blockIdx.x % heads;
    const size_t base = (size_t)blockIdx.x * kDh * n;   // the 16 channels of a head are consecutive rows
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    kt += (size_t)h * period;   // lag u at u mod period, |u| < n
    auto value = [&](int lag) { return lag < n && lag > -n ? __ldg(kt + (lag < 0 ? period + lag : lag)) : 0.f; };
    bool earlier = false;       // a lag below zero is not zero
    for (int u = 1 + tid; u < n; u += kThreads) earlier |= value(-u) != 0.f;
    // copy p (p = 0, 1): the kernel value of a lag lies at np + 14 + p - lag
    for (int i = tid; i < kc; i += kThreads) {
        const int lag = np + 14 - i;
        const float a = value(lag);
        ks[i] = a;
        if (i + 1 < kc) ks[kc + i + 1] = a;
    }
    if (tid == 0) ks[kc] = 0.f;   // (lag np + 15)
    const __nv_bfloat16* src[3] = {X1 + base, X2 + base, V + base};
    if (n % 8 == 0) {   // 16-byte pieces never straddle a row
        constexpr int kW = kThreads / 32, kR = 3 * kDh / kW / 2;   // rows per warp, in two rounds of loads in flight
        for (int c = lane * 8; c < n; c += 256)
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                uint4 v[kR];
#pragma unroll
                for (int q = 0; q < kR; ++q) {
                    const int r = warp + kW * (z * kR + q);   // row of the three tensors one after the other
                    v[q] = __ldg(reinterpret_cast<const uint4*>((r < kDh ? src[0] : r < 2 * kDh ? src[1] : src[2]) + (size_t)(r % kDh) * n + c));
                }
#pragma unroll
                for (int q = 0; q < kR; ++q) *reinterpret_cast<uint4*>(xs1 + (warp + kW * (z * kR + q)) * ld + c) = v[q];
            }
        if (np != n && tid < 3 * kDh) *reinterpret_cast<uint4*>(xs1 + tid * ld + n) = make_uint4(0u, 0u, 0u, 0u);
    } else {
        for (int r = warp; r < kDh; r += kThreads / 32)
            for (int c = lane; c < np; c += 32)
#pragma unroll
                for (int q = 0; q < 3; ++q) xs1[q * kDh * ld + r * ld + c] = c < n ? src[q][(size_t)r * n + c] : __float2bfloat16_rn(0.f);
    }
    earlier = __syncthreads_or(earlier);
    const int m = lane >> 3, r8 = lane & 7, g = lane >> 2, c2 = 2 * (lane & 3);
    // ldmatrix row addresses: A of the scores (X1, transposed on load), B of the scores (X2, transposed), A of the output (V)
    const uint32_t a1 = smem_addr(xs1 + ((m >> 1) * 8 + r8) * ld + (m & 1) * 8);
    const uint32_t b2 = smem_addr(xs2 + ((m & 1) * 8 + r8) * ld + (m >> 1) * 8);
    const uint32_t av = smem_addr(vs + ((m & 1) * 8 + r8) * ld + (m >> 1) * 8);
    const float* kp = ks + (g & 1) * kc + np + 14 + (g & 1) - g + c2;   // lag g - c2; minus the tile distance
    const int tiles = np / 16, groups = (tiles + T - 1) / T, nw = kThreads / 32;
    const int front = nw * ((groups + 2 * nw - 1) / (2 * nw));   // the first half of a warp's groups in order, the second from the far end:
    auto walk = [&](auto both) {   // (two tiles at a time, both sides of the diagonal: a loop of its own, so that the other stays as it is)
        for (int it = warp; it < groups; it += nw) {                 // every warp gets as many short ones as long ones
            const int t0 = T * (it < front ? it : groups - 1 - (it - front));
            uint32_t fa[T][4];
#pragma unroll
            for (int z = 0; z < T; ++z) ldsm4t(fa[z], a1 + min(t0 + z, tiles - 1) * 32);   // (past the last tile: that tile again, its products are not stored)
            float o[T][2][4] = {};
            uint32_t fb[4] = {}, fv[4] = {};   // the tile si of X2 and of V
            auto tile = [&](int z, float2 k0, float2 k8, float2 km) {   // the kernel at lags u, u + 8, u - 8 and the one below each
                float s0[4] = {}, s1[4] = {};
                mma(s0, fa[z], fb[0], fb[1]);
                mma(s1, fa[z], fb[2], fb[3]);
                mma(o[z][0], fv, weigh(s0[0], s0[1], k0), weigh(s1[0], s1[1], km));
                mma(o[z][1], fv, weigh(s0[2], s0[3], k8), weigh(s1[2], s1[3], k0));
            };
            auto kernel = [&](const float* q) { return *reinterpret_cast<const float2*>(q); };
            if constexpr (T == 1) {
                for (int si = 0; si <= t0; ++si) {
                    const float* kq = kp - (t0 - si) * 16;
                    ldsm4t(fb, b2 + si * 32);
                    ldsm4(fv, av + si * 32);
                    tile(0, kernel(kq), kernel(kq - 8), kernel(kq + 8));
                }
            } else {
                const float* kq = kp;   // one tile further away with every step down in s: what was 8 above is then 8 below
                float2 k0 = kernel(kq), k8 = kernel(kq - 8), km = kernel(kq + 8);
                if (t0 + 1 < tiles) {
                    ldsm4t(fb, b2 + t0 * 32 + 32);
                    ldsm4(fv, av + t0 * 32 + 32);
                    tile(1, k0, k8, km);
                }
                for (int si = t0; si >= 0; --si) {
                    kq -= 16;
                    const float2 n0 = kernel(kq), n8 = kernel(kq - 8);
                    ldsm4t(fb, b2 + si * 32);
                    ldsm4(fv, av + si * 32);
                    tile(0, k0, k8, km);
                    tile(1, n0, n8, k8);
                    km = k8;
                    k0 = n0;
                    k8 = n8;
                }
            }
            if constexpr (T == 1) {
                if (earlier) {
                    auto below = [&](int lag) { return lag > -n ? __ldg(kt + period + lag) : 0.f; };   // (every lag of these tiles is below zero)
                    auto pair = [&](int lag) { return make_float2(below(lag), below(lag - 1)); };
                    float2 k8 = pair(g - c2 - 8);
#pragma unroll 1
                    for (int d = 16; d < np - 16 * t0; d += 16) {
                        const float2 k0 = pair(g - c2 - d), km = pair(g - c2 - d - 8);
                        ldsm4t(fb, b2 + t0 * 32 + 2 * d);
                        ldsm4(fv, av + t0 * 32 + 2 * d);
                        tile(0, k0, k8, km);
                        k8 = km;   // (what was 8 below is 8 above a step later)
                    }
                }
            } else if constexpr (decltype(both)::value) {
                auto pair = [&](int lag) { return make_float2(value(lag), value(lag - 1)); };
                int u = g - c2 - 16;
                float2 k0 = pair(u), k8 = pair(u + 8), km = pair(u - 8), l0 = {}, l8 = {}, lm = {};   // this step's, the step's before: one tile further away
#pragma unroll 1
                for (int si = t0 + 1; si < tiles; ++si) {
                    u -= 16;
                    const float2 n0 = pair(u), nm = pair(u - 8);   // the next step's, on their way while this one is multiplied
                    ldsm4t(fb, b2 + si * 32);
                    ldsm4(fv, av + si * 32);
                    tile(0, k0, k8, km);
                    if (si > t0 + 1) tile(1, l0, l8, lm);
                    l0 = k0;
                    l8 = k8;
                    lm = km;
                    k8 = km;
                    k0 = n0;
                    km = nm;
                }
            }
            __syncwarp();   // these tiles' columns of X1 are read by this warp alone, above: the result takes their place
#pragma unroll
            for (int z = 0; z < T; ++z) {
                if (t0 + z >= tiles) break;
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    *reinterpret_cast<uint32_t*>(xs1 + g * ld + (t0 + z) * 16 + x * 8 + c2) = bf2(o[z][x][0], o[z][x][1]);
                    *reinterpret_cast<uint32_t*>(xs1 + (g + 8) * ld + (t0 + z) * 16 + x * 8 + c2) = bf2(o[z][x][2], o[z][x][3]);
                }
            }
        }
    };
    if (T > 1 && earlier)
        walk(std::true_type{});
    else
        walk(std::false_type{});
    __syncthreads();
    if (n % 8 == 0) {
        for (int r = warp; r < kDh; r += kThreads / 32)
            for (int c = lane * 8; c < n; c += 256)
                *reinterpret_cast<uint4*>(O + base + (size_t)r * n + c) = *reinterpret_cast<const uint4*>(xs1 + r * ld + c);
    } else {
        for (int r = warp; r < kDh; r += kThreads / 32)
            for (int c = lane; c < n; c += 32) O[base + (size_t)r * n + c] = xs1[r * ld + c];
    }
}

bool covered(const m2_plan* pl, int64_t n, int64_t d, int64_t dh) {
    return pl->dtype == M2_BF16 && m2f::covered(pl) && dh == kDh && d % kDh == 0 && n > 0 && n <= kMaxN;
}

int32_t heads_fwd(const m2_plan* pl, const void* X1, const void* X2, const void* V, const float* kt, int64_t period, void* O, int64_t B, int64_t d,
                  int64_t n, cudaStream_t stream) {
    const int64_t blocks = B * (d / kDh);
    if (blocks == 0) return M2_OK;
    if (blocks > 0x7fffffffLL) return M2_ERR_UNSUPPORTED;
    const int smem = smem_bytes((int)n);
    // Two tiles at a time halve the fragments and kernel values read per tile pair and leave a warp half as many groups.  Layer of d = 768, us,
    // one tile and two: n = 1024, [8] (batch) 204.6 and 178.9, [1] 82.6 and 86.7; n = 512 [32] 261 and 242, [1] 66.2 and 59.9; 320 [8] 75.6 and 71.0;
    // 256 [32] 89.4 and 85.7, [16] 61.9 and 60.6, [8] 49.1 and 49.8; 208 [24] 70.0 and 69.9, [8] 46.0 and 46.8.  Rows beyond 512, layers of some widths by
    // blocks: n = 1024 [48] 87.8 and 90.5, [64] 77.5 and 82.4, [72] 90.1 and 86.1, [144] 102.8 and 97.4; 1000 [48] 87.6 and 92.0, [64] 78.5 and 83.8; 640 [48] 72.1 and
    // 74.3, [64] 66.0 and 70.1, [192] 87.8 and 86.4.  (The kernel alone is faster with two at [48] as well, 24.1 and 20.3 for 1024;
    // why the layers are not was not found.  [8] and [24] would gain, 67.5 and 54.4, 86.6 and 83.4.)
    const bool pairs = n > 512 ? blocks > 64 : n > 256 || (n > 224 && blocks >= 768);
    const int threads = pairs && n <= 256 ? 128 : 256;
    auto kern = !pairs ? heads_kernel<256, 1> : n <= 256 ? heads_kernel<128, 2> : heads_kernel<256, 2>;
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(kMaxN)) != cudaSuccess)
        return M2_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, (const __nv_bfloat16*)X1, (const __nv_bfloat16*)X2, (const __nv_bfloat16*)V, kt, (int)period,
                           (__nv_bfloat16*)O, (int)(d / kDh), (int)n) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2h
