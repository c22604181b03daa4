// Kernel spectrum and kernel gradient of the fp32 transform path (fft_conv.cu has the convolution).
#include "fft_conv.h"
#include "fft_pass.cuh"

namespace m2f {

// k_f of one channel per row: the forward half alone, scaled by 1 / N
template <class C, bool HALF>
__global__ void __launch_bounds__(C::THREADS, min_blocks<C>())
    fft_spectrum_kernel(const float* __restrict__ k, float4* __restrict__ kf, float4* __restrict__ kfu, float* __restrict__ kt,
                        float sgn, const float4* __restrict__ tab, int H, int n) {
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = threadIdx.x / C::TP, t = threadIdx.x % C::TP;
    const long long h = (long long)blockIdx.x * C::ROWS + r;
    const bool live = h < H;
    float* sr = smem + r * C::ROWF + (r & 1) * C::PAR;
    float* si = sr + C::SMEM_FLOATS;
    u64 re[16], im[16];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // rows of k are only as aligned as n floats make them; a pair needs 8 bytes
    load_row<C, float, HALF>(re, k + h * n, t, n, (n & 1) == 0 && (reinterpret_cast<uintptr_t>(k) & 7) == 0, live);
    unroll<16>([&](auto j) { im[j.v] = 0ull; });
    if (kt != nullptr && live) {   // a thread's 32 values, eight on their way together (spectrum, forward and both gradients of [32][768][512]: 72.9 us one by one, 69.7 in eights)
#pragma unroll
        for (int g = 0; g < 32; g += 8) {
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int i = t + (g + q) * C::TP;
                v[q] = i < n ? __ldg(k + h * n + i) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) kt[h * C::N + t + (g + q) * C::TP] = v[q];
        }
    }
    forward<C, HALF>(re, im, sr, si, tab, t, r);
    if (!live) return;
    const u64 sc = dup2(1.0f / (float)C::N);
    float4* out = kf + h * (C::N / 2) + t;
    unroll<16>([&](auto s) {
        constexpr int p = brev<4>(s.v);
        re[p] = mul2(re[p], sc);
        im[p] = mul2(im[p], sc);
        out[s.v * C::TP] = make_float4(lo(re[p]), hi(re[p]), lo(im[p]), hi(im[p]));
    });
    if constexpr (C::N == 512) {
        // thread t = q1 holds the frequencies q1 + 16 q2, q2 in the low halves of slots 0 .. 15, then in the high ones: k1 = q1 + 16 c,
        // k2 = 2 q, 2 q + 1 is q2 = 4 q + c, 4 q + 2 + c
        if (kfu != nullptr) {
            float4* priv = kfu + h * 256 + t;
            unroll<16>([&](auto s) {
                constexpr int q = s.v / 2, c = s.v % 2, qa = 4 * q + c, qb = qa + 2, pa = brev<4>(qa & 15), pb = brev<4>(qb & 15);
                priv[q * 32 + c * 16] = qa < 16 ? make_float4(lo(re[pa]), lo(re[pb]), sgn * lo(im[pa]), sgn * lo(im[pb]))
                                                : make_float4(hi(re[pa]), hi(re[pb]), sgn * hi(im[pa]), sgn * hi(im[pb]));
            });
        }
    }
}

// Values of `share` neighbouring rows of threads added in order: value (s, t) of a channel = the sum over its rows' threads t; share * TP
// threads share the work.  all: 16 float4 per thread of the block; other rows may still be reading it on return
template <class C>
__device__ __forceinline__ void add_shares(u64* re, u64* im, float4* all, int share, int r, int t) {
    float4* own = all + threadIdx.x;
    __syncthreads();
    unroll<16>([&](auto s) { own[s.v * C::THREADS] = make_float4(lo(re[s.v]), hi(re[s.v]), lo(im[s.v]), hi(im[s.v])); });
    __syncthreads();
    const int first = (r / share) * share * C::TP, lid = threadIdx.x - first, step = share * C::TP;
    for (int v = lid; v < 16 * C::TP; v += step) {
        float4* p = all + (v / C::TP) * C::THREADS + first + v % C::TP;
        float4 a = *p;
        for (int q = 1; q < share; ++q) {
            const float4 w = p[q * C::TP];
            a.x += w.x;
            a.y += w.y;
            a.z += w.z;
            a.w += w.w;
        }
        *p = a;
    }
    __syncthreads();
    unroll<16>([&](auto s) {
        const float4 a = all[s.v * C::THREADS + first + t];
        re[s.v] = pk(a.x, a.y);
        im[s.v] = pk(a.z, a.w);
    });
}

// the inverse half alone, of the sum of `parts` spectra: scale times the real part of the first n positions.  `share` rows of threads
// (a power of two) take the parts of one channel in turn, as in fft_wgrad_kernel: a part is a round trip to memory, and few channels with
// many parts waited for one after the other (x, g [4096][1][256], the whole gradient: 136 us with 256 parts added by one row of threads,
// 30 by eight).  both: rows of 2 n values, the first n positions and the last n (2 n <= N), where what is below 2^-20 of the row's largest
// value -- the transforms' rounding, if the kernel has no such lags -- is written as zero.
template <class C, bool HALF>
__global__ void __launch_bounds__(C::THREADS, min_blocks<C>())
    fft_time_kernel(const float4* __restrict__ kf, int parts, float scale, float* __restrict__ kt, const float4* __restrict__ tab, int H,
                    int n, int share, int both) {
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = threadIdx.x / C::TP, t = threadIdx.x % C::TP;
    const long long h = (long long)blockIdx.x * (C::ROWS / share) + r / share;
    const bool live = h < H;
    float* sr = smem + r * C::ROWF + (r & 1) * C::PAR;
    float* si = sr + C::SMEM_FLOATS;
    u64 re[16], im[16];
    const float4* in = kf + ((long long)(r % share) * H + (live ? h : 0)) * (C::N / 2) + t;   // (share <= parts)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    unroll<16>([&](auto s) {
        constexpr int p = brev<4>(s.v);
        const float4 w = in[s.v * C::TP];
        re[p] = pk(w.x, w.y);
        im[p] = pk(w.z, w.w);
    });
#pragma unroll 1
    for (int q = r % share + share; q < parts; q += share) {
        in += (long long)share * H * (C::N / 2);
        unroll<16>([&](auto s) {
            constexpr int p = brev<4>(s.v);
            const float4 w = in[s.v * C::TP];
            re[p] = add2(re[p], pk(w.x, w.y));
            im[p] = add2(im[p], pk(w.z, w.w));
        });
    }
    if constexpr (C::ROWS > 1) {
        static_assert(2 * C::SMEM_FLOATS * 4 >= C::THREADS * 256, "the rows' values fit where the transform exchanges its digits");
        if (share > 1) {
            add_shares<C>(re, im, reinterpret_cast<float4*>(smem), share, r, t);
            __syncthreads();
        }
    }
    const u64 sc = dup2(scale);
    unroll<16>([&](auto s) {
        re[s.v] = mul2(re[s.v], sc);
        im[s.v] = mul2(im[s.v], sc);
    });
    inverse<C, HALF>(re, im, sr, si, tab, t, r);
    if (!HALF && both) {   // (one launch-wide choice: the threads of a row meet)
        uint32_t top, same;
        pair_tops<C, false>(re, re, reinterpret_cast<uint32_t*>(smem + 2 * C::SMEM_FLOATS) + r * scale_words<C>(), t, r, top, same);
        const float least = __uint_as_float(top) * 0x1p-20f;
        auto put = [&](int i, float v) {
            if (i < n) kt[h * 2 * n + i] = v;
            else if (i >= C::N - n) kt[h * 2 * n + i - (C::N - 2 * n)] = fabsf(v) <= least ? 0.f : v;
        };
        if (live && r % share == 0)
            unroll<16>([&](auto q) {
                constexpr int p = brev<4>(q.v), STEP = C::N / C::R1;
                put(C::R1 == 16 ? q.v * STEP + 2 * t : q.v * STEP + t, lo(re[p]));
                put(C::R1 == 16 ? q.v * STEP + 2 * t + 1 : (q.v + 16) * STEP + t, hi(re[p]));
            });
        return;
    }
    store_row<C, float, HALF>(re, kt + h * n, t, n, (n & 1) == 0, live && r % share == 0);
}

// dk[h] = Re F^-1( sum over row pairs of conj(F z) (.) F w ) / N with z = x_a + i x_b, w = g_a + i g_b: the real part of the product's
// inverse is corr(x_a, g_a) + corr(x_b, g_b).  `share` rows of threads (a power of two) take the pairs of one channel in turn; a row's
// sum stays in registers, F z waits in shared memory in the thread's own slots, and the rows' sums are added in order at the end.
// (One row per channel left most SMs idle at short lengths: bf16 [64][768][256] 319 -> 35 us, [32][768][512] 176 -> 35 us with the
// loads of a row in flight together, too.)
// Three transforms follow one another and a pair's cross terms cancel, so differences are taken directly where the other kernels save two
// of eight FMAs (fft_core.cuh): in the inverse and with constant factors everywhere, with variable factors at N = 256, where the dense
// stages of a 16 x 16 plan are the most accurate.  Distance from the exact gradient, fp32: N = 4096 causal 2.46e-7 without, 2.39e-7 so (16 x 16 x 16
// dense stages: 2.40e-7), N = 256 causal 2.02e-7 and 1.90e-7 (1.92e-7); x, g [4][768][2048] 36.9 and 37.5 us.
template <class C>
constexpr int kGradDirect = C::N == 256 ? 2 : 1;
template <class C>
constexpr int wgrad_blocks() { return C::THREADS == 128 ? 2 : 1; }
template <class C, typename IO, bool HALF>
__global__ void __launch_bounds__(C::THREADS, wgrad_blocks<C>())
    fft_wgrad_kernel(const IO* __restrict__ x, const IO* __restrict__ g, float* __restrict__ dk, const float4* __restrict__ tab, int B, int H,
                     int n, int share) {
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = threadIdx.x / C::TP, t = threadIdx.x % C::TP;
    const long long h = (long long)blockIdx.x * (C::ROWS / share) + r / share;
    const bool live = h < H, vec = (n & 1) == 0;
    float* sr = smem + r * C::ROWF + (r & 1) * C::PAR;
    float* si = sr + C::SMEM_FLOATS;
    float4* zall = reinterpret_cast<float4*>(smem + 2 * C::SMEM_FLOATS);
    float4* zs = zall + threadIdx.x;
    uint32_t* slot = reinterpret_cast<uint32_t*>(zall + C::THREADS * 16) + r * scale_words<C>();
    u64 re[16], im[16], ar[16], ai[16];
    unroll<16>([&](auto s) { ar[s.v] = ai[s.v] = 0ull; });
    asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
    for (int b0 = 0; b0 < B; b0 += 2 * share) {   // (every row of threads takes every step: the barriers may span several rows)
        const int b = b0 + 2 * (r % share);
        const bool has_a = live && b < B, has_b = live && b + 1 < B;
        const long long oa = has_a ? ((long long)b * H + h) * n : 0, ob = oa + (long long)H * n;
        load_row<C, IO, HALF>(re, x + oa, t, n, vec, has_a);
        load_row<C, IO, HALF>(im, x + ob, t, n, vec, has_b);
        uint32_t ta, tb;
        int ea, eb;   // x / 2^e and 2^e g: the cross terms of a pair are then no larger than the pair's share of the sum
        pair_tops<C, HALF>(re, im, slot, t, r, ta, tb);
        pair_exponents(ta, tb, ea, eb);
        scale_row<HALF>(re, scale_down(ea));
        scale_row<HALF>(im, scale_down(eb));
        forward<C, HALF, kGradDirect<C>>(re, im, sr, si, tab, t, r);
        unroll<16>([&](auto s) { zs[s.v * C::THREADS] = make_float4(lo(re[s.v]), hi(re[s.v]), lo(im[s.v]), hi(im[s.v])); });
        load_row<C, IO, HALF>(re, g + oa, t, n, vec, has_a);
        load_row<C, IO, HALF>(im, g + ob, t, n, vec, has_b);
        scale_row<HALF>(re, scale_up(ea));
        scale_row<HALF>(im, scale_up(eb));
        row_sync<C>(r);
        forward<C, HALF, kGradDirect<C>>(re, im, sr, si, tab, t, r);
        unroll<16>([&](auto s) {   // += conj(z) w
            const float4 z = zs[s.v * C::THREADS];
            const u64 zr = pk(z.x, z.y), zi = pk(z.z, z.w);
            ar[s.v] = fma2(zr, re[s.v], fma2(zi, im[s.v], ar[s.v]));
            ai[s.v] = fma2(zr, im[s.v], fma2(neg2(zi), re[s.v], ai[s.v]));
        });
        row_sync<C>(r);
    }
    if (C::ROWS > 1 && share > 1) add_shares<C>(ar, ai, zall, share, r, t);
    inverse<C, HALF, 2>(ar, ai, sr, si, tab, t, r);
    const u64 sc = dup2(1.0f / (float)C::N);
    unroll<16>([&](auto s) { ar[s.v] = mul2(ar[s.v], sc); });
    store_row<C, float, HALF>(ar, dk + h * n, t, n, vec, live && r % share == 0);
}

template <class C>
constexpr int wgrad_smem() { return conv_smem<C>() + C::THREADS * 16 * 16; }

cudaError_t prepare_gradients(const m2_plan* pl) {
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        cudaError_t e = allow_smem(fft_spectrum_kernel<C, false>, conv_smem<C>());
        if (e == cudaSuccess) e = allow_smem(fft_spectrum_kernel<C, true>, conv_smem<C>());
        if (e == cudaSuccess) e = allow_smem(fft_time_kernel<C, false>, conv_smem<C>());
        if (e == cudaSuccess) e = allow_smem(fft_time_kernel<C, true>, conv_smem<C>());
        if constexpr (C::N <= 8192) {
            auto io = [&](auto z) {
                using IO = decltype(z);
                if (e == cudaSuccess) e = allow_smem(fft_wgrad_kernel<C, IO, false>, wgrad_smem<C>());
                if (e == cudaSuccess) e = allow_smem(fft_wgrad_kernel<C, IO, true>, wgrad_smem<C>());
            };
            if (pl->dtype == M2_BF16) io(__nv_bfloat16());
            else io(float());
        }
        return e;
    });
}

cudaError_t spectrum(const m2_plan* pl, const float* k, int64_t H, int64_t n, void* kf, void* kfu, float* kt, cudaStream_t stream) {
    if (H == 0) return cudaSuccess;
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        const unsigned grid = (unsigned)((H + C::ROWS - 1) / C::ROWS);
        const float sgn = pl->sign >= 0 ? 1.0f : -1.0f;
        auto go = [&](auto half) {
            return launch_early(fft_spectrum_kernel<C, decltype(half)::v != 0>, grid, C::THREADS, conv_smem<C>(), stream, k, (float4*)kf,
                                (float4*)kfu, kt, sgn, (const float4*)pl->d_fft, (int)H, (int)n);
        };
        return 2 * n <= C::N ? go(Ic<1>{}) : go(Ic<0>{});
    });
}

cudaError_t time_kernel(const m2_plan* pl, const void* kf, int parts, float scale, int64_t H, int64_t n, bool both, float* kt,
                        cudaStream_t stream) {
    if (H == 0) return cudaSuccess;
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        int share = 1;   // rows of a block per channel: no more than there are parts
        while (share < C::ROWS && 2 * share <= parts) share *= 2;
        const int64_t per_block = C::ROWS / share;
        const unsigned grid = (unsigned)((H + per_block - 1) / per_block);
        auto go = [&](auto half) {
            return launch_early(fft_time_kernel<C, decltype(half)::v != 0>, grid, C::THREADS, conv_smem<C>(), stream, (const float4*)kf, parts,
                                scale, kt, (const float4*)pl->d_fft, (int)H, (int)n, share, (int)both);
        };
        return 2 * n <= C::N && !both ? go(Ic<1>{}) : go(Ic<0>{});
    });
}

cudaError_t wgrad(const m2_plan* pl, const void* x, const void* g, float* dk, int64_t B, int64_t H, int64_t n, bool causal,
                  cudaStream_t stream) {
    if (H == 0) return cudaSuccess;
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        if constexpr (C::N > 8192) {
            return cudaErrorInvalidValue;
        } else {
            int share = 1;   // rows of a block per channel: no more than there are pairs
            while (share < C::ROWS && 2 * share < B) share *= 2;
            const int64_t per_block = C::ROWS / share;
            const unsigned grid = (unsigned)((H + per_block - 1) / per_block);
            auto go = [&](auto z, auto half) {
                using IO = decltype(z);
                return launch_early(fft_wgrad_kernel<C, IO, decltype(half)::v != 0>, grid, C::THREADS, wgrad_smem<C>(), stream, (const IO*)x,
                                    (const IO*)g, dk, (const float4*)pl->d_fft, (int)B, (int)H, (int)n, share);
            };
            if (pl->dtype == M2_BF16) return causal ? go(__nv_bfloat16(), Ic<1>{}) : go(__nv_bfloat16(), Ic<0>{});
            return causal ? go(float(), Ic<1>{}) : go(float(), Ic<0>{});
        }
    });
}

}  // namespace m2f
