// The passes of fft_core.cuh put together for one row of threads (load, forward transform, inverse transform, store) and the dispatch
// over the row length; included by the files that instantiate kernels from them.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fft_core.cuh"
#include "m2_plan.h"

namespace m2f {

// A pair of neighbouring values as it lies in memory (raw), and as two fp32 values.  The loads of a row are written down apart from
// the conversions so that all of them are in flight together (bf16 x[4][768][4096]: 39.5 -> 31.0 us; kernel gradient 71 -> 45 us).
template <typename IO>
struct Io;
template <>
struct Io<float> {
    typedef u64 raw2;
    typedef float raw;
    static __device__ __forceinline__ u64 cvt2(raw2 w) { return w; }
    static __device__ __forceinline__ float cvt(raw w) { return w; }
    static __device__ __forceinline__ void st2(float* p, u64 v) { *reinterpret_cast<u64*>(p) = v; }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <>
struct Io<__nv_bfloat16> {
    typedef uint32_t raw2;
    typedef unsigned short raw;
    static __device__ __forceinline__ u64 cvt2(raw2 w) { return pk(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)); }
    static __device__ __forceinline__ float cvt(raw w) { return __uint_as_float((uint32_t)w << 16); }
    static __device__ __forceinline__ void st2(__nv_bfloat16* p, u64 v) {
        *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(lo(v), hi(v));
    }
    static __device__ __forceinline__ void st(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// threads of one row meet; rows that fit in a warp need no block-wide barrier
template <class C>
__device__ __forceinline__ void row_sync(int r) {
    if constexpr (C::TP <= 32) __syncwarp();
    else if constexpr (C::ROWS == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(r + 1), "n"(C::TP) : "memory");
}

// input digit n1 of the thread's first-pass columns; positions >= n, or a row that is not there, read as zero.  vec: the row's length
// is even, so a pair of neighbouring positions is one aligned load and lies on one side of n
template <class C, typename IO, bool HALF>
__device__ __forceinline__ void load_row(u64* v, const IO* row, int t, int n, bool vec, bool have) {
    constexpr int JN = HALF ? C::R1 / 2 : C::R1;
    constexpr int STEP = C::N / C::R1;
    typedef typename Io<IO>::raw2 raw2;
    typedef typename Io<IO>::raw raw;
    if (sizeof(IO) == 4 && !have) {   // fp32 loads go straight into place; the branch keeps the two rows' address registers apart
        unroll<(C::R1 == 16 ? JN : JN / 2)>([&](auto j) { v[j.v] = 0ull; });
        return;
    }
    const int lim = sizeof(IO) == 4 || have ? n : 0;   // bf16: no branch, both rows' loads are in flight together
    if (C::R1 == 16 && vec) {
        raw2 w[16];
        unroll<JN>([&](auto j) {
            const int i = j.v * STEP + 2 * t;
            w[j.v] = 0;
            if (i < lim) w[j.v] = __ldg(reinterpret_cast<const raw2*>(row + i));
        });
        unroll<JN>([&](auto j) { v[j.v] = Io<IO>::cvt2(w[j.v]); });
    } else {
        raw w[32];
        constexpr int L = C::R1 == 16 ? 2 * JN : JN;
        // A whole row needs no bound per load: with 32 of them per row and four rows the bounds kept bf16 loads of the kernel gradient
        // from being in flight together (N = 1024, 16 rows of 768 channels: 76.9 us with
        // them, 39.2 without; fp32 40; the convolution 29.6 -> 23.7, causal 23.0 -> 20.5).
        if (sizeof(IO) == 2 && C::R1 == 32 && lim >= L * STEP)
            unroll<L>([&](auto j) { w[j.v] = __ldg(reinterpret_cast<const raw*>(row + j.v * STEP + t)); });
        else
            unroll<L>([&](auto j) {
                const int i = C::R1 == 16 ? (j.v / 2) * STEP + 2 * t + (j.v & 1) : j.v * STEP + t;
                w[j.v] = 0;
                if (i < lim) w[j.v] = __ldg(reinterpret_cast<const raw*>(row + i));
            });
        unroll<L / 2>([&](auto j) { v[j.v] = pk(Io<IO>::cvt(w[2 * j.v]), Io<IO>::cvt(w[2 * j.v + 1])); });
    }
}
// output digit n1 = q in slot brev(q) (R1 = 32: q and q + 16)
template <class C, typename IO, bool HALF>
__device__ __forceinline__ void store_row(const u64* v, IO* row, int t, int n, bool vec, bool have) {
    constexpr int JN = HALF ? C::R1 / 2 : C::R1;
    constexpr int STEP = C::N / C::R1;
    if (sizeof(IO) == 4 && !have) return;
    const int lim = sizeof(IO) == 4 || have ? n : 0;
    if constexpr (C::R1 == 16) {
        unroll<JN>([&](auto q) {
            constexpr int p = brev<4>(q.v);
            const int i = q.v * STEP + 2 * t;
            if (vec) {
                if (i < lim) Io<IO>::st2(row + i, v[p]);
            } else {
                if (i < lim) Io<IO>::st(row + i, lo(v[p]));
                if (i + 1 < lim) Io<IO>::st(row + i + 1, hi(v[p]));
            }
        });
    } else {
        unroll<16>([&](auto q) {
            constexpr int p = brev<4>(q.v);
            const int i = q.v * STEP + t;
            if (i < lim) Io<IO>::st(row + i, lo(v[p]));
            if (!HALF && i + 16 * STEP < lim) Io<IO>::st(row + i + 16 * STEP, hi(v[p]));
        });
    }
}

// ---- two real rows as one complex row ----
// The rounding error of a transform is relative to the norm of the complex row, and a value that is not finite reaches all of it, so the
// two rows are made alike first: each is multiplied by a power of two, which is exact and is taken back when the row leaves (without that
// a row beside one 1e4 times as large is about 1e-3 off).  The first row's brings its largest magnitude to [1, 2), the second's comes
// nearest to the same, so that rows of one distribution keep the ratio they have (with both in [1, 2) they ended up a factor of two apart
// now and then, and the errors 5 % larger).  One B200, without and with the factors: bf16 x[8][768][2000] 44.9 and 46.3 us,
// [16][768][1024] 21.3 and 23.4, fp32 [4][768][2048] 26.2 and 26.9.
template <class C>
__host__ __device__ constexpr int scale_words() { return 2 * (C::TP > 32 ? C::TP / 32 + 1 : 1); }   // per row pair: its warps' maxima, the factors
template <class C>
__host__ __device__ constexpr int scale_bytes() { return (C::ROWS * scale_words<C>() * 4 + 15) / 16 * 16; }
constexpr uint32_t kInfBits = 0x7f800000u;

// largest magnitudes of the pair's rows as bits, NaN above infinity above everything else; each thread brings its part of both.  Ends
// with a barrier of the row's threads where they are in several warps
template <class C, bool HALF>
__device__ __forceinline__ void pair_tops(const u64* re, const u64* im, uint32_t* slot, int t, int r, uint32_t& ta, uint32_t& tb) {
    auto top = [](const u64* v) {
        float m = 0.f;
        unroll<(HALF ? 8 : 16)>([&](auto j) { asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(lo(v[j.v])), "f"(hi(v[j.v]))); });
        return __float_as_uint(m);
    };
    ta = top(re);
    tb = top(im);
    if constexpr (C::TP >= 32) {
        ta = __reduce_max_sync(0xffffffffu, ta);
        tb = __reduce_max_sync(0xffffffffu, tb);
    } else {
#pragma unroll
        for (int o = C::TP / 2; o > 0; o /= 2) {
            ta = max(ta, __shfl_xor_sync(0xffffffffu, ta, o));
            tb = max(tb, __shfl_xor_sync(0xffffffffu, tb, o));
        }
    }
    if constexpr (C::TP > 32) {
        if (t % 32 == 0) {
            slot[t / 32 * 2] = ta;
            slot[t / 32 * 2 + 1] = tb;
        }
        row_sync<C>(r);
#pragma unroll
        for (int w = 0; w < C::TP / 32; ++w) {
            ta = max(ta, slot[2 * w]);
            tb = max(tb, slot[2 * w + 1]);
        }
    }
}
// exponent fields of the rows' powers of two (the power and its inverse are normal numbers); a row that is not finite counts as zeros
__device__ __forceinline__ void pair_exponents(uint32_t ta, uint32_t tb, int& ea, int& eb) {
    const int a = ta >= kInfBits ? 0 : (int)ta, b = tb >= kInfBits ? 0 : (int)tb;
    ea = min(max(a >> 23, 1), 253);
    eb = min(max(ea - ((a - b + (1 << 22)) >> 23), 1), 253);   // the bits of a float are its logarithm, nearly
}
__device__ __forceinline__ float scale_up(int e) { return __uint_as_float((uint32_t)e << 23); }
__device__ __forceinline__ float scale_down(int e) { return __uint_as_float((uint32_t)(254 - e) << 23); }
template <bool HALF>
__device__ __forceinline__ void scale_row(u64* v, float f) {   // as load_row leaves it
    const u64 w = dup2(f);
    unroll<(HALF ? 8 : 16)>([&](auto j) { v[j.v] = mul2(v[j.v], w); });
}
// Makes a pair's rows alike for a convolution.  A row with a value that is not finite takes no part (zeros) and leaves as NaN, a row of
// zeros leaves as zeros.
template <class C, bool HALF>
__device__ __forceinline__ void balance_pair(u64* re, u64* im, uint32_t* slot, int t, int r) {
    uint32_t ta, tb;
    pair_tops<C, HALF>(re, im, slot, t, r, ta, tb);
    int ea, eb;
    pair_exponents(ta, tb, ea, eb);
    auto one = [&](u64* v, uint32_t top, int e, uint32_t* back) {
        if (top >= kInfBits) unroll<(HALF ? 8 : 16)>([&](auto j) { v[j.v] = 0ull; });
        else scale_row<HALF>(v, scale_down(e));
        if (t == 0) *back = top >= kInfBits ? 0x7fffffffu : top == 0 ? 0u : __float_as_uint(scale_up(e));
    };
    one(re, ta, ea, slot + scale_words<C>() - 2);
    one(im, tb, eb, slot + scale_words<C>() - 1);
}
// (the row's threads have met since)
template <class C>
__device__ __forceinline__ void unbalance_pair(u64* re, u64* im, const uint32_t* slot) {
    const u64 fa = dup2(__uint_as_float(slot[scale_words<C>() - 2])), fb = dup2(__uint_as_float(slot[scale_words<C>() - 1]));
    unroll<16>([&](auto s) {
        re[s.v] = mul2(re[s.v], fa);
        im[s.v] = mul2(im[s.v], fb);
    });
}

// registers (input digit of the first pass) -> registers (output of the last digit: q in slot brev(q); R = 32: q, q + 16).
// The row's shared memory must be free on entry; afterwards other threads may still be reading it.
template <class C, bool HALF, int P = 0>
__device__ __forceinline__ void forward(u64* re, u64* im, float* sr, float* si, const float4* __restrict__ tab, int t, int r) {
    fft_first<C, HALF, P>(re, im);
    put_first<C>(re, im, sr, si, t);
    row_sync<C>(r);
    if constexpr (C::THREE) {
        auto m1 = [&](int c, int j) { return mid1<C>(t, c, j); };
        auto m2 = [&](int c, int j) { return mid2<C>(t, c, j); };
        get_cols<C::R2>(re, im, sr, si, m1);
        row_sync<C>(r);
        fft_tw<C::R2, P>(re, im, tab + Tab<C>::F2 + t / C::R3, Tab<C>::K2);
        put_cols<C::R2>(re, im, sr, si, m2);
        row_sync<C>(r);
    }
    get_cols<C::RL>(re, im, sr, si, [&](int c, int j) { return last2<C>(t, c, j); });
    fft_tw<C::RL, P>(re, im, tab + Tab<C>::FL + t, C::TP);
}
// registers (as forward leaves them) -> registers (output digit n1 of the first-pass columns); re and im swapped by the caller's
// choice of names: the inverse transform is the forward one on (im, re)
template <class C, bool HALF, int P = 0>
__device__ __forceinline__ void inverse(u64* re, u64* im, float* sr, float* si, const float4* __restrict__ tab, int t, int r) {
    if constexpr (C::RL == 16) fft_packed<16, false, true, false, false, P>(im, re, nullptr, 0);
    else fft32_dif<P>(im, re);
    put_cols_natural<C::RL>(re, im, sr, si, [&](int c, int j) { return last2<C>(t, c, j); });   // the thread's own columns: in place
    row_sync<C>(r);
    if constexpr (C::THREE) {
        auto m1 = [&](int c, int j) { return mid1<C>(t, c, j); };
        auto m2 = [&](int c, int j) { return mid2<C>(t, c, j); };
        get_cols<C::R2>(re, im, sr, si, m2);
        row_sync<C>(r);
        fft_tw<C::R2, P>(im, re, tab + Tab<C>::I2 + t % C::R3, C::R3);
        put_cols<C::R2>(re, im, sr, si, m1);
        row_sync<C>(r);
    }
    if constexpr (C::R1 == 16) {
        unroll<16>([&](auto j) {
            if constexpr (C::THREE) {
                re[j.v] = *reinterpret_cast<const u64*>(sr + j.v * C::S1 + 2 * t);
                im[j.v] = *reinterpret_cast<const u64*>(si + j.v * C::S1 + 2 * t);
            } else {
                re[j.v] = pk(sr[j.v * C::S1 + 2 * t], sr[j.v * C::S1 + 2 * t + 1]);
                im[j.v] = pk(si[j.v * C::S1 + 2 * t], si[j.v * C::S1 + 2 * t + 1]);
            }
        });
        fft_packed<16, true, false, false, HALF, P>(im, re, tab + Tab<C>::I1 + t, C::TP);
    } else {
        get_cols<C::R1>(re, im, sr, si, [&](int, int j) { return j * C::S1 + t; });
        fft32_eo<true, false, HALF, P>(im, re, tab + Tab<C>::I1 + t, C::TP);
    }
}

template <class C>
constexpr int min_blocks() { return C::THREADS == 128 ? 4 : C::THREADS == 256 ? 2 : 1; }

// ---- host side -----------------------------------------------------------------------------------------------------------------

inline int log2_exact(int64_t N) {
    for (int l = 8; l <= 14; ++l)
        if (N == (int64_t)1 << l) return l;
    return 0;
}
// calls f(Cfg<log2 N>{})
template <class F>
cudaError_t dispatch(int64_t N, F&& f) {
    switch (log2_exact(N)) {
        case 8: return f(Cfg<8>{});
        case 9: return f(Cfg<9>{});
        case 10: return f(Cfg<10>{});
        case 11: return f(Cfg<11>{});
        case 12: return f(Cfg<12>{});
        case 13: return f(Cfg<13>{});
        case 14: return f(Cfg<14>{});
    }
    return cudaErrorInvalidValue;
}

template <class C>
constexpr int conv_smem() { return 2 * C::SMEM_FLOATS * 4 + scale_bytes<C>(); }
template <class K>
cudaError_t allow_smem(K kern, int bytes) {
    return bytes > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) : cudaSuccess;
}

// launch that lets the blocks start while the previous kernel's last ones still run (they wait before they touch its results)
template <class... P, class... A>
cudaError_t launch_early(void (*kern)(P...), unsigned grid, int threads, int smem, cudaStream_t stream, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace m2f
