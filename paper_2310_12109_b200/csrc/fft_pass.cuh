// The passes of fft_core.cuh put together for one row of threads (load, forward transform, inverse transform, store) and the dispatch
// over the row length; included by the files that instantiate kernels from them.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fft_core.cuh"
#include "m2_plan.h"

namespace m2f {

template <typename IO>
struct Io;
template <>
struct Io<float> {
    static __device__ __forceinline__ u64 ld2(const float* p) { return *reinterpret_cast<const u64*>(p); }
    static __device__ __forceinline__ float ld(const float* p) { return *p; }
    static __device__ __forceinline__ void st2(float* p, u64 v) { *reinterpret_cast<u64*>(p) = v; }
    static __device__ __forceinline__ void st(float* p, float v) { *p = v; }
};
template <>
struct Io<__nv_bfloat16> {
    static __device__ __forceinline__ u64 ld2(const __nv_bfloat16* p) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
        return pk(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
    static __device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
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

// input digit n1 of the thread's first-pass columns; positions >= n and a missing row read as zero.  vec: n is even, so a pair of
// neighbouring positions is one aligned load and lies on one side of n
template <class C, typename IO, bool HALF>
__device__ __forceinline__ void load_row(u64* v, const IO* row, int t, int n, bool vec) {
    constexpr int JN = HALF ? C::R1 / 2 : C::R1;
    constexpr int STEP = C::N / C::R1;
    if constexpr (C::R1 == 16) {
        if (row == nullptr) {
            unroll<JN>([&](auto j) { v[j.v] = 0ull; });
        } else if (vec) {
            unroll<JN>([&](auto j) {
                const int i = j.v * STEP + 2 * t;
                v[j.v] = i < n ? Io<IO>::ld2(row + i) : 0ull;
            });
        } else {
            unroll<JN>([&](auto j) {
                const int i = j.v * STEP + 2 * t;
                v[j.v] = pk(i < n ? Io<IO>::ld(row + i) : 0.f, i + 1 < n ? Io<IO>::ld(row + i + 1) : 0.f);
            });
        }
    } else {
        unroll<JN / 2>([&](auto m) {
            const int i = 2 * m.v * STEP + t;
            v[m.v] = row == nullptr ? 0ull : pk(i < n ? Io<IO>::ld(row + i) : 0.f, i + STEP < n ? Io<IO>::ld(row + i + STEP) : 0.f);
        });
    }
}
// output digit n1 = q in slot brev(q) (R1 = 32: q and q + 16)
template <class C, typename IO, bool HALF>
__device__ __forceinline__ void store_row(const u64* v, IO* row, int t, int n, bool vec) {
    constexpr int JN = HALF ? C::R1 / 2 : C::R1;
    constexpr int STEP = C::N / C::R1;
    if (row == nullptr) return;
    if constexpr (C::R1 == 16) {
        unroll<JN>([&](auto q) {
            constexpr int p = brev<4>(q.v);
            const int i = q.v * STEP + 2 * t;
            if (vec) {
                if (i < n) Io<IO>::st2(row + i, v[p]);
            } else {
                if (i < n) Io<IO>::st(row + i, lo(v[p]));
                if (i + 1 < n) Io<IO>::st(row + i + 1, hi(v[p]));
            }
        });
    } else {
        unroll<16>([&](auto q) {
            constexpr int p = brev<4>(q.v);
            const int i = q.v * STEP + t;
            if (i < n) Io<IO>::st(row + i, lo(v[p]));
            if (!HALF && i + 16 * STEP < n) Io<IO>::st(row + i + 16 * STEP, hi(v[p]));
        });
    }
}

// registers (input digit of the first pass) -> registers (output of the last digit: q in slot brev(q); R = 32: q, q + 16).
// The row's shared memory must be free on entry; afterwards other threads may still be reading it.
template <class C, bool HALF>
__device__ __forceinline__ void forward(u64* re, u64* im, float* sr, float* si, const float4* __restrict__ tab, int t, int r) {
    fft_first<C, HALF>(re, im);
    put_first<C>(re, im, sr, si, t);
    row_sync<C>(r);
    if constexpr (C::THREE) {
        auto m1 = [&](int c, int j) { return mid1<C>(t, c, j); };
        auto m2 = [&](int c, int j) { return mid2<C>(t, c, j); };
        get_cols<C::R2>(re, im, sr, si, m1);
        row_sync<C>(r);
        fft_tw<C::R2>(re, im, tab + Tab<C>::F2 + t / C::R3, Tab<C>::K2);
        put_cols<C::R2>(re, im, sr, si, m2);
        row_sync<C>(r);
    }
    get_cols<C::RL>(re, im, sr, si, [&](int c, int j) { return last2<C>(t, c, j); });
    fft_tw<C::RL>(re, im, tab + Tab<C>::FL + t, C::TP);
}
// registers (as forward leaves them) -> registers (output digit n1 of the first-pass columns); re and im swapped by the caller's
// choice of names: the inverse transform is the forward one on (im, re)
template <class C, bool HALF>
__device__ __forceinline__ void inverse(u64* re, u64* im, float* sr, float* si, const float4* __restrict__ tab, int t, int r) {
    if constexpr (C::RL == 16) fft_packed<16, false, true, false, false>(im, re, nullptr, 0);
    else fft32_dif(im, re);
    put_cols_natural<C::RL>(re, im, sr, si, [&](int c, int j) { return last2<C>(t, c, j); });   // the thread's own columns: in place
    row_sync<C>(r);
    if constexpr (C::THREE) {
        auto m1 = [&](int c, int j) { return mid1<C>(t, c, j); };
        auto m2 = [&](int c, int j) { return mid2<C>(t, c, j); };
        get_cols<C::R2>(re, im, sr, si, m2);
        row_sync<C>(r);
        fft_tw<C::R2>(im, re, tab + Tab<C>::I2 + t % C::R3, C::R3);
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
        fft_packed<16, true, false, false, HALF>(im, re, tab + Tab<C>::I1 + t, C::TP);
    } else {
        get_cols<C::R1>(re, im, sr, si, [&](int, int j) { return j * C::S1 + t; });
        fft32_eo<true, false, HALF>(im, re, tab + Tab<C>::I1 + t, C::TP);
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
constexpr int conv_smem() { return 2 * C::SMEM_FLOATS * 4; }
template <class K>
cudaError_t allow_smem(K kern, int bytes) {
    return bytes > 48 * 1024 ? cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) : cudaSuccess;
}

}  // namespace m2f
