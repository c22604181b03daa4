// Register-level pieces of the fp32 transform kernels (fft_conv.cu): packed fp32x2 arithmetic, transforms of 8, 16 and 32 points
// held in one thread's registers, and the thread <-> column <-> shared-memory maps of a factorisation N = R1 R2 (R3).
//
// A transform of N points is N = R1 R2 R3 (or R1 R2) digits contracted one after the other, the same order-p factorisation of F_N
// that the plan uses (Corollary "DFT is M"), with digits of 8 to 32 so that a digit fits in a thread's registers:
//   n = (n1 R2 + n2) R3 + n3,  k = q1 + R1 q2 + R1 R2 q3.
// A thread always holds 32 complex points, in 16 slots of two packed values: two columns of 16, four columns of 8 (two sets of
// two), or one column of 32.  Two values of one kind share a 64-bit register pair, so every add and FMA is one f32x2 instruction:
// the FP32 pipe does the same 128 lanes per cycle either way, but packed instructions leave half of the issue slots to the
// shared-memory traffic of the digit exchanges, which is the other thing these kernels are bound by.
//
// Twiddles multiply the INPUTS of a contraction, x[j] -> x[j] w^j with a per-column base w.  They are folded into the butterflies
// (decimation in time): X[q], X[q + S/2] = E[q] +- (w^{R/S} W_S^q) O[q] costs six FMAs whatever the factor is, and since
// W_S^{S/4} = i a 16-point column needs only eight factors.  The sign of the exponent is always +; the inverse transform is the
// forward one with the roles of real and imaginary part exchanged.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

#define M2_HD __host__ __device__ __forceinline__

namespace m2f {

typedef unsigned long long u64;

M2_HD u64 pk(float lo, float hi) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
#else
    uint32_t a, b;
    memcpy(&a, &lo, 4);
    memcpy(&b, &hi, 4);
    return ((u64)b << 32) | a;
#endif
}
M2_HD void upk(u64 v, float& lo, float& hi) {
#ifdef __CUDA_ARCH__
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
#else
    uint32_t a = (uint32_t)v, b = (uint32_t)(v >> 32);
    memcpy(&lo, &a, 4);
    memcpy(&hi, &b, 4);
#endif
}
M2_HD float lo(u64 v) { float a, b; upk(v, a, b); return a; }
M2_HD float hi(u64 v) { float a, b; upk(v, a, b); return b; }
M2_HD u64 fma2(u64 a, u64 b, u64 c) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
#else
    return pk(lo(a) * lo(b) + lo(c), hi(a) * hi(b) + hi(c));
#endif
}
M2_HD u64 mul2(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
#else
    return pk(lo(a) * lo(b), hi(a) * hi(b));
#endif
}
M2_HD u64 add2(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
#else
    return pk(lo(a) + lo(b), hi(a) + hi(b));
#endif
}
M2_HD u64 sub2(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
#else
    return pk(lo(a) - lo(b), hi(a) - hi(b));
#endif
}
M2_HD u64 neg2(u64 a) { return pk(-lo(a), -hi(a)); }   // (becomes a source modifier of the instruction that reads it)
M2_HD u64 dup2(float a) { return pk(a, a); }

// W_32^q = exp(+2 pi i q / 32), q < 8 (the others follow by symmetry)
template <int Q>
struct W32 {
    static constexpr double c[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708, 0.70710678118654752440,
                                    0.55557023301960222474, 0.38268343236508977173, 0.19509032201612826785, 0.0};
    static constexpr int q = Q & 31;
    static constexpr int oct = q <= 8 ? q : q <= 16 ? 16 - q : q <= 24 ? q - 16 : 32 - q;
    static constexpr double re = (q <= 8 || q >= 24) ? c[oct] : -c[oct];
    static constexpr double im = q <= 16 ? c[8 - oct] : -c[8 - oct];
};

template <int LOG>
M2_HD constexpr int brev(int v) {
    int r = 0;
    for (int i = 0; i < LOG; ++i) r |= ((v >> i) & 1) << (LOG - 1 - i);
    return r;
}

// compile-time loop: f(std::integral_constant<int, I>) for I = 0 .. N - 1
template <int I>
struct Ic {
    static constexpr int v = I;
    M2_HD constexpr operator int() const { return I; }
};
template <int I, int N, class F>
M2_HD void unroll_from(F&& f) {
    if constexpr (I < N) {
        f(Ic<I>{});
        unroll_from<I + 1, N>(f);
    }
}
template <int N, class F>
M2_HD void unroll(F&& f) { unroll_from<0, N>(f); }

// o+- = a +- w b in place (a, b <- o+, o-); ROT: the factor is i w.  PLUS_ONLY: o- is not needed.
// P: o- as 2 a - o+, two FMAs and one rounding more (0), or directly, four: with constant factors (1), with all (2).
template <bool ROT, bool PLUS_ONLY, int P>
M2_HD void bfly(u64& ar, u64& ai, u64& br, u64& bi, u64 wr, u64 wi) {
    const u64 two = dup2(2.0f);
    u64 pr, pi;
    if (!ROT) {
        pr = fma2(wr, br, fma2(neg2(wi), bi, ar));
        pi = fma2(wr, bi, fma2(wi, br, ai));
    } else {
        pr = fma2(neg2(wi), br, fma2(neg2(wr), bi, ar));
        pi = fma2(wr, br, fma2(neg2(wi), bi, ai));
    }
    if constexpr (!PLUS_ONLY && P >= 2) {
        u64 mr, mi;
        if (!ROT) {
            mr = fma2(neg2(wr), br, fma2(wi, bi, ar));
            mi = fma2(neg2(wr), bi, fma2(neg2(wi), br, ai));
        } else {
            mr = fma2(wi, br, fma2(wr, bi, ar));
            mi = fma2(neg2(wr), br, fma2(wi, bi, ai));
        }
        br = mr;
        bi = mi;
    } else if constexpr (!PLUS_ONLY) {
        br = fma2(two, ar, neg2(pr));
        bi = fma2(two, ai, neg2(pi));
    }
    ar = pr;
    ai = pi;
}
// the same with the constant factor W_32^Q
template <int Q, bool PLUS_ONLY, int P>
M2_HD void bfly_const(u64& ar, u64& ai, u64& br, u64& bi) {
    if constexpr ((Q & 31) == 0) {
        const u64 pr = add2(ar, br), pi = add2(ai, bi);
        if (!PLUS_ONLY) {
            br = sub2(ar, br);
            bi = sub2(ai, bi);
        }
        ar = pr;
        ai = pi;
    } else if constexpr ((Q & 31) == 8) {   // factor i
        const u64 pr = sub2(ar, bi), pi = add2(ai, br);
        if (!PLUS_ONLY) {
            const u64 mr = add2(ar, bi);
            bi = sub2(ai, br);
            br = mr;
        }
        ar = pr;
        ai = pi;
    } else {
        const float c = (float)W32<Q>::re, s = (float)W32<Q>::im;
        const u64 pr = fma2(dup2(c), br, fma2(dup2(-s), bi, ar)), pi = fma2(dup2(c), bi, fma2(dup2(s), br, ai));
        if constexpr (!PLUS_ONLY && P >= 1) {
            const u64 mr = fma2(dup2(-c), br, fma2(dup2(s), bi, ar)), mi = fma2(dup2(-c), bi, fma2(dup2(-s), br, ai));
            br = mr;
            bi = mi;
        } else if constexpr (!PLUS_ONLY) {
            br = fma2(dup2(2.0f), ar, neg2(pr));
            bi = fma2(dup2(2.0f), ai, neg2(pi));
        }
        ar = pr;
        ai = pi;
    }
}

// R-point transform (R = 8, 16) of packed columns in slots base .. base + R - 1.
//   TW: factors from tw[v * stride] = (re0, re1, im0, im1), v = 0: S = 2, 1: S = 4, 2, 3: S = 8, 4 .. 7: S = 16
//   BRIN = false: input j in slot j, output q in slot brev(q); BRIN = true: input j in slot brev(j), output q in slot q
//   HALF_IN: inputs j >= R / 2 are zero (their slots are not read); HALF_OUT: only outputs q < R / 2 are computed
template <int R, bool TW, bool BRIN, bool HALF_IN, bool HALF_OUT, int P>
M2_HD void fft_packed(u64* re, u64* im, const float4* tw, int stride) {
    constexpr int LOG = R == 16 ? 4 : 3;
    auto slot = [](int pos) constexpr { return BRIN ? pos : brev<LOG>(pos); };
    unroll<LOG>([&](auto lv) {
        constexpr int S = 2 << lv.v, HS = S / 2;
        [[maybe_unused]] constexpr int V0 = S == 2 ? 0 : S / 4;       // first factor of this level
        if constexpr (S == 2 && HALF_IN) {                             // the second input of every butterfly is zero
            unroll<R / 2>([&](auto b) {
                constexpr int p0 = slot(2 * b.v), p1 = slot(2 * b.v + 1);
                re[p1] = re[p0];
                im[p1] = im[p0];
            });
        } else {
            unroll<HS>([&](auto q) {
                constexpr bool rot = S >= 4 && q.v >= S / 4;
                constexpr bool plus = HALF_OUT && S == R;
                [[maybe_unused]] u64 wr = 0, wi = 0;
                if constexpr (TW) {
                    const float4 w = tw[(V0 + (rot ? q.v - S / 4 : q.v)) * stride];
                    wr = pk(w.x, w.y);
                    wi = pk(w.z, w.w);
                }
                unroll<R / S>([&](auto b) {
                    constexpr int p0 = slot(b.v * S + q.v), p1 = slot(b.v * S + q.v + HS);
                    if constexpr (TW) bfly<rot, plus, P>(re[p0], im[p0], re[p1], im[p1], wr, wi);
                    else bfly_const<q.v * (32 / S), plus, P>(re[p0], im[p0], re[p1], im[p1]);
                });
            });
        }
    });
}

// 32-point transform of one column: input slot m = (x[2m], x[2m+1]), output q, q + 16 in slot brev(q) = (X[q], X[q+16]).
//   TW: tw[v * stride], v < 8: the 16-point factors of base w^2, both halves equal; v = 8 + q / 2: (re, im) of w W_32^q for q, q + 1
template <bool TW, bool HALF_IN, bool HALF_OUT, int P>
M2_HD void fft32_eo(u64* re, u64* im, const float4* tw, int stride) {
    fft_packed<16, TW, false, HALF_IN, false, P>(re, im, tw, stride);
    unroll<16>([&](auto q) {   // last level: even part E[q] in the low half, odd part O[q] in the high half
        constexpr int p = brev<4>(q.v);
        constexpr bool rot = q.v >= 8;
        float er, orr, ei, oi, wr, wi;
        upk(re[p], er, orr);
        upk(im[p], ei, oi);
        if constexpr (TW) {
            const float4 w = tw[(8 + (q.v & 7) / 2) * stride];
            const float cr = (q.v & 1) ? w.z : w.x, ci = (q.v & 1) ? w.w : w.y;
            wr = rot ? -ci : cr;
            wi = rot ? cr : ci;
        } else {
            wr = (float)W32<q.v>::re;
            wi = (float)W32<q.v>::im;
        }
        const float pr = fmaf(wr, orr, fmaf(-wi, oi, er)), pi = fmaf(wr, oi, fmaf(wi, orr, ei));
        float mr = 0.f, mi = 0.f;
        if constexpr (!HALF_OUT) {
            mr = P >= (TW ? 2 : 1) ? fmaf(-wr, orr, fmaf(wi, oi, er)) : fmaf(2.0f, er, -pr);
            mi = P >= (TW ? 2 : 1) ? fmaf(-wr, oi, fmaf(-wi, orr, ei)) : fmaf(2.0f, ei, -pi);
        }
        re[p] = pk(pr, mr);
        im[p] = pk(pi, mi);
    });
}

// 32-point transform without factors that takes what fft32_eo left: input slot brev(j) = (x[j], x[j+16]), output slot m = (X[2m], X[2m+1])
template <int P>
M2_HD void fft32_dif(u64* re, u64* im) {
    unroll<16>([&](auto j) {
        constexpr int p = brev<4>(j.v);
        float ar, br, ai, bi;
        upk(re[p], ar, br);
        upk(im[p], ai, bi);
        const float ur = ar + br, ui = ai + bi, vr = ar - br, vi = ai - bi;
        if constexpr (j.v == 0) {
            re[p] = pk(ur, vr);
            im[p] = pk(ui, vi);
        } else if constexpr (j.v == 8) {
            re[p] = pk(ur, -vi);
            im[p] = pk(ui, vr);
        } else {
            const float c = (float)W32<j.v>::re, s = (float)W32<j.v>::im;
            re[p] = pk(ur, fmaf(c, vr, -s * vi));
            im[p] = pk(ui, fmaf(c, vi, s * vr));
        }
    });
    fft_packed<16, false, true, false, false, P>(re, im, nullptr, 0);
}

// ---- factorisations ------------------------------------------------------------------------------------------------------------
// TP = N / 32 threads work on one complex row; ROWS rows share a block of 128 threads (more for long rows).  Shared-memory maps, in
// floats, real and imaginary parts in separate arrays (strides chosen so that every access pattern below is free of bank conflicts,
// checked exhaustively; the one exception is the last digit of N = 2048, two-way):
//   two digits     Z[q1][n2] at q1 S1 + n2
//   three digits   Z[q1][n2][n3] at q1 S1 + n2 R3 + n3 after the first digit, Z[q1][n3][q2] at q1 S2 + n3 ST + q2 after the second
template <int LOGN>
struct Cfg;
#define M2_FFT_CFG(LOGN_, R1_, R2_, R3_, S1_, S2_, ST_, ROWF_, PAR_)                                                                  \
    template <>                                                                                                                       \
    struct Cfg<LOGN_> {                                                                                                               \
        static constexpr int N = 1 << LOGN_, R1 = R1_, R2 = R2_, R3 = R3_, TP = N / 32, S1 = S1_, S2 = S2_, ST = ST_, ROWF = ROWF_,   \
                             PAR = PAR_, THREADS = TP < 128 ? 128 : TP, ROWS = THREADS / TP;                                          \
        static constexpr bool THREE = R3 > 1;                                                                                         \
        static constexpr int RL = THREE ? R3 : R2;   /* the digit contracted last */                                                  \
        static constexpr int SMEM_FLOATS = ROWS * ROWF + 4;                                                                           \
        static_assert(R1 * R2 * R3 == N, "digits");                                                                                   \
    };
M2_FFT_CFG(8, 16, 16, 1, 18, 0, 0, 296, 1)
M2_FFT_CFG(9, 16, 32, 1, 34, 0, 0, 544, 1)
M2_FFT_CFG(10, 32, 32, 1, 33, 0, 0, 1056, 0)
M2_FFT_CFG(11, 16, 8, 16, 144, 144, 9, 2304, 0)
M2_FFT_CFG(12, 16, 16, 16, 272, 272, 17, 4352, 0)
M2_FFT_CFG(13, 16, 16, 32, 512, 560, 17, 8960, 0)
M2_FFT_CFG(14, 16, 32, 32, 1024, 1056, 33, 16896, 0)
#undef M2_FFT_CFG

// Twiddle tables of one plan, one after the other in device memory; offsets in float4.  entries(R): factors a column of R needs.
M2_HD constexpr int tw_entries(int R) { return R == 32 ? 12 : 8; }   // (R = 8: four for each of the two sets of columns)
template <class C>
struct Tab {
    static constexpr int K2 = C::THREE ? C::R1 / (32 / C::R2) : 0;                   // forward middle digit: one row per q1 (of the first column)
    static constexpr int F2 = 0;
    static constexpr int FL = F2 + (C::THREE ? tw_entries(C::R2) * K2 : 0);        // forward last digit: one row per thread
    static constexpr int I2 = FL + tw_entries(C::RL) * C::TP;                      // inverse middle digit: one row per n3
    static constexpr int I1 = I2 + (C::THREE ? tw_entries(C::R2) * C::R3 : 0);     // inverse first digit: one row per thread
    static constexpr int END = I1 + tw_entries(C::R1) * C::TP;
};

// column c of thread t (c < 32 / R) in each pass, as the exponent e of its twiddle base omega_N^e ... used by the table builder
template <class C>
M2_HD int col_last(int t, int c) {   // forward last digit: q1 + R1 q2
    if (C::THREE) return (t / C::R2 + c * (C::R1 / (32 / C::R3))) + C::R1 * (t % C::R2);
    return t + c * (C::R1 / (32 / C::R2));
}
template <class C>
M2_HD int col_first(int t, int c) { return C::R1 == 16 ? 2 * t + c : t; }   // first digit: n mod N / R1

// where the spectrum value of frequency k lives: float index within a channel's 2 N floats
template <class C>
M2_HD int spec_index(int k, bool imag) {
    const int q1 = k % C::R1, q2 = (k / C::R1) % C::R2, q3 = k / (C::R1 * C::R2);
    const int ql = C::THREE ? q3 : q2;
    int t, s, half;
    if (C::RL == 16) {
        const int g = C::R1 / 2;   // the thread's two columns are q1 and q1 + R1 / 2
        half = q1 / g;
        t = C::THREE ? (q1 % g) * C::R2 + q2 : q1 % g;
        s = ql;
    } else {
        t = C::THREE ? q1 * C::R2 + q2 : q1;
        half = ql / 16;
        s = ql % 16;
    }
    return (s * C::TP + t) * 4 + (imag ? 2 : 0) + half;
}
M2_HD int spec_index_any(int logn, int k, bool imag) {
    switch (logn) {
        case 8: return spec_index<Cfg<8>>(k, imag);
        case 9: return spec_index<Cfg<9>>(k, imag);
        case 10: return spec_index<Cfg<10>>(k, imag);
        case 11: return spec_index<Cfg<11>>(k, imag);
        case 12: return spec_index<Cfg<12>>(k, imag);
        case 13: return spec_index<Cfg<13>>(k, imag);
        default: return spec_index<Cfg<14>>(k, imag);
    }
}

// ---- passes of one thread (t < TP) on its row's shared-memory arrays sr, si ------------------------------------------------------
// Each pass reads its columns from the registers or from shared memory, contracts one digit, and leaves the result in registers
// (fft_*) or writes it (put_*); the caller places the barriers.

template <class C, bool HALF_IN, int P>
M2_HD void fft_first(u64* re, u64* im) {   // registers: input digit n1 of the thread's columns
    if constexpr (C::R1 == 16) fft_packed<16, false, false, HALF_IN, false, P>(re, im, nullptr, 0);
    else fft32_eo<false, HALF_IN, false, P>(re, im, nullptr, 0);
}
template <class C>
M2_HD void put_first(const u64* re, const u64* im, float* sr, float* si, int t) {
    unroll<16>([&](auto q) {
        constexpr int p = brev<4>(q.v);
        if constexpr (C::R1 == 16 && C::THREE) {   // two neighbouring columns: one 64-bit store
            *reinterpret_cast<u64*>(sr + q.v * C::S1 + 2 * t) = re[p];
            *reinterpret_cast<u64*>(si + q.v * C::S1 + 2 * t) = im[p];
        } else if constexpr (C::R1 == 16) {
            sr[q.v * C::S1 + 2 * t] = lo(re[p]);
            sr[q.v * C::S1 + 2 * t + 1] = hi(re[p]);
            si[q.v * C::S1 + 2 * t] = lo(im[p]);
            si[q.v * C::S1 + 2 * t + 1] = hi(im[p]);
        } else {
            sr[q.v * C::S1 + t] = lo(re[p]);
            sr[(q.v + 16) * C::S1 + t] = hi(re[p]);
            si[q.v * C::S1 + t] = lo(im[p]);
            si[(q.v + 16) * C::S1 + t] = hi(im[p]);
        }
    });
}

// address of element j of column c of the middle pass: layout 1 (before / after the inverse) and layout 2
template <class C>
M2_HD int mid1(int t, int c, int j) { return (t / C::R3 + c * (C::R1 / (32 / C::R2))) * C::S1 + j * C::R3 + t % C::R3; }
template <class C>
M2_HD int mid2(int t, int c, int j) { return (t / C::R3 + c * (C::R1 / (32 / C::R2))) * C::S2 + (t % C::R3) * C::ST + j; }
// the same for the last digit
template <class C>
M2_HD int last2(int t, int c, int j) {
    if (C::THREE) return (t / C::R2 + c * (C::R1 / (32 / C::R3))) * C::S2 + j * C::ST + t % C::R2;
    return (t + c * (C::R1 / (32 / C::R2))) * C::S1 + j;
}

// ADDR(t, c, j) -> registers: R = 8: slots 8 (c / 2) + j, half c % 2; R = 16: slot j, half c; R = 32: slot j / 2, half j % 2
template <int R, class A>
M2_HD void get_cols(u64* re, u64* im, const float* sr, const float* si, A addr) {
    unroll<16>([&](auto s) {
        constexpr int j0 = R == 32 ? 2 * s.v : R == 16 ? s.v : s.v % 8, c0 = R == 8 ? 2 * (s.v / 8) : 0;
        constexpr int j1 = R == 32 ? j0 + 1 : j0, c1 = R == 32 ? 0 : c0 + 1;
        const int a0 = addr(c0, j0), a1 = addr(c1, j1);
        re[s.v] = pk(sr[a0], sr[a1]);
        im[s.v] = pk(si[a0], si[a1]);
    });
}
// outputs of a BRIN = false transform (R = 32: of fft32_eo): R = 8, 16: output q in slot brev(q); R = 32: q, q + 16 in slot brev(q)
template <int R, class A>
M2_HD void put_cols(const u64* re, const u64* im, float* sr, float* si, A addr) {
    unroll<16>([&](auto s) {
        constexpr int q0 = R == 8 ? brev<3>(s.v % 8) : brev<4>(s.v), c0 = R == 8 ? 2 * (s.v / 8) : 0;
        constexpr int q1 = R == 32 ? q0 + 16 : q0, c1 = R == 32 ? 0 : c0 + 1;
        const int a0 = addr(c0, q0), a1 = addr(c1, q1);
        sr[a0] = lo(re[s.v]);
        sr[a1] = hi(re[s.v]);
        si[a0] = lo(im[s.v]);
        si[a1] = hi(im[s.v]);
    });
}
// outputs in natural slots: R = 16: q in slot q; R = 32 (fft32_dif): 2m, 2m + 1 in slot m
template <int R, class A>
M2_HD void put_cols_natural(const u64* re, const u64* im, float* sr, float* si, A addr) {
    unroll<16>([&](auto s) {
        constexpr int q0 = R == 32 ? 2 * s.v : s.v, q1 = R == 32 ? q0 + 1 : q0, c1 = R == 32 ? 0 : 1;
        const int a0 = addr(0, q0), a1 = addr(c1, q1);
        sr[a0] = lo(re[s.v]);
        sr[a1] = hi(re[s.v]);
        si[a0] = lo(im[s.v]);
        si[a1] = hi(im[s.v]);
    });
}
template <int R, int P>
M2_HD void fft_tw(u64* re, u64* im, const float4* tw, int stride) {
    if constexpr (R == 8) {
        fft_packed<8, true, false, false, false, P>(re, im, tw, stride);
        fft_packed<8, true, false, false, false, P>(re + 8, im + 8, tw + 4 * stride, stride);
    } else if constexpr (R == 16) {
        fft_packed<16, true, false, false, false, P>(re, im, tw, stride);
    } else {
        fft32_eo<true, false, false, P>(re, im, tw, stride);
    }
}

}  // namespace m2f
