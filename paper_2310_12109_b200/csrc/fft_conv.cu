// Convolution in fp32 (fft_grad.cu: kernel spectrum, and the kernel gradient up to 8192 points) for every plan whose length is a power
// of two from 256 to 16384: the fp32 path, and the bf16 shapes the tensor-core kernels do not cover.  A complex row (two real batch rows
// of one channel: the kernel is real, so F^-1(k_f (.) F(x_a + i x_b)) = y_a + i y_b; balance_pair keeps them apart) stays in registers
// and shared memory from the load to the store; fft_core.cuh has the transforms.
//
// What bounds it: shared-memory wavefronts (64 KB each way per digit exchange of a 4096-point row), packed FP32 and the loads and stores
// of a row that nothing overlaps within its block; with 126 registers four blocks of 128 threads share an SM.  bf16 x[8][768][2000], N =
// 4096, one B200: 46 us (0.2 of the roof: its bytes take 9.8 us; the wavefronts alone would take 22 us), 66 % of the load/store data
// pipe, 49 % of the FMA pipe, 46 % of the issue slots, DRAM 12 %; 6034 us for the kernel before it, which contracted each 64-wide
// digit as a dense product in shared memory with a sincos per element.  fp32 x[1][4][256]: 18.4 -> 6.5 us per call, one launch and the
// host's way to it.
#include <atomic>
#include <cmath>
#include <vector>

#include "fft_conv.h"
#include "fft_pass.cuh"

namespace m2f {

template <class C, typename IO, bool HALF>
__global__ void __launch_bounds__(C::THREADS, min_blocks<C>())
    fft_conv_kernel(const IO* __restrict__ x, const float4* __restrict__ kf, IO* __restrict__ y, const float4* __restrict__ tab, int B, int H,
                    int n, long long npairs, int kf_group) {
    extern __shared__ __align__(16) float smem[];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = threadIdx.x / C::TP, t = threadIdx.x % C::TP;
    const long long pair = (long long)blockIdx.x * C::ROWS + r;
    const int per_h = (B + 1) / 2;
    const bool vec = (n & 1) == 0;
    const bool live = pair < npairs;
    const int h = live ? (int)(pair / per_h) : 0, b = live ? 2 * (int)(pair % per_h) : 0;
    float* sr = smem + r * C::ROWF + (r & 1) * C::PAR;
    float* si = sr + C::SMEM_FLOATS;
    const long long oa = ((long long)b * H + h) * n, ob = oa + (long long)H * n;
    const bool has_b = live && b + 1 < B;
    u64 re[16], im[16];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    load_row<C, IO, HALF>(re, x + oa, t, n, vec, live);
    load_row<C, IO, HALF>(im, x + ob, t, n, vec, has_b);
    uint32_t* slot = reinterpret_cast<uint32_t*>(smem + 2 * C::SMEM_FLOATS) + r * scale_words<C>();
    balance_pair<C, HALF>(re, im, slot, t, r);
    forward<C, HALF>(re, im, sr, si, tab, t, r);
    const float4* kr = kf + (long long)(h / kf_group) * (C::N / 2) + t;
    unroll<16>([&](auto s) {
        constexpr int p = brev<4>(s.v);
        const float4 w = kr[s.v * C::TP];
        const u64 wr = pk(w.x, w.y), wi = pk(w.z, w.w);
        const u64 pr = fma2(wr, re[p], neg2(mul2(wi, im[p])));
        im[p] = fma2(wr, im[p], mul2(wi, re[p]));
        re[p] = pr;
    });
    inverse<C, HALF>(re, im, sr, si, tab, t, r);
    unbalance_pair<C>(re, im, slot);
    store_row<C, IO, HALF>(re, y + oa, t, n, vec, live);
    store_row<C, IO, HALF>(im, y + ob, t, n, vec, has_b);
}

// ---- host side -----------------------------------------------------------------------------------------------------------------

bool covered(const m2_plan* pl) { return pl->d_fft != nullptr; }
int spectrum_order(const m2_plan* pl) { return covered(pl) ? log2_exact(pl->N) : 0; }

// rows x entries factors: entry v of row i at tab[off + v * rows + i]; expo(i, c) = exponent of omega_N of the base of column c
template <class E>
static void fill(std::vector<float4>& tab, int off, int N, int R, int rows, E expo, const std::vector<double2>& root) {
    auto w = [&](long long e) { return root[(size_t)(e % N)]; };
    for (int i = 0; i < rows; ++i) {
        auto put = [&](int v, double2 a, double2 b) { tab[off + v * rows + i] = make_float4((float)a.x, (float)b.x, (float)a.y, (float)b.y); };
        auto levels = [&](int v0, int RR, long long ea, long long eb) {
            int v = v0;
            for (int S = 2; S <= RR; S *= 2)
                for (int q = 0; q < (S == 2 ? 1 : S / 4); ++q, ++v)
                    put(v, w(ea * (RR / S) + (long long)q * (N / S)), w(eb * (RR / S) + (long long)q * (N / S)));
        };
        if (R == 8) {
            levels(0, 8, expo(i, 0), expo(i, 1));
            levels(4, 8, expo(i, 2), expo(i, 3));
        } else if (R == 16) {
            levels(0, 16, expo(i, 0), expo(i, 1));
        } else {
            const long long e = expo(i, 0);
            levels(0, 16, 2 * e, 2 * e);
            for (int q = 0; q < 8; q += 2) {
                const double2 a = w(e + (long long)q * (N / 32)), b = w(e + (long long)(q + 1) * (N / 32));
                tab[off + (8 + q / 2) * rows + i] = make_float4((float)a.x, (float)a.y, (float)b.x, (float)b.y);
            }
        }
    }
}

template <class C>
static std::vector<float4> build_tab() {
    std::vector<double2> root(C::N);
    for (int j = 0; j < C::N; ++j) {
        const double a = 2.0 * M_PI * (double)j / (double)C::N;
        root[j] = make_double2(std::cos(a), std::sin(a));
    }
    std::vector<float4> tab(Tab<C>::END);
    if (C::THREE) {
        fill(tab, Tab<C>::F2, C::N, C::R2, Tab<C>::K2, [](int i, int c) { return (long long)(i + c * Tab<C>::K2) * C::R3; }, root);
        fill(tab, Tab<C>::I2, C::N, C::R2, C::R3, [](int i, int) { return (long long)i * C::R1; }, root);
    }
    fill(tab, Tab<C>::FL, C::N, C::RL, C::TP, [](int i, int c) { return (long long)col_last<C>(i, c); }, root);
    fill(tab, Tab<C>::I1, C::N, C::R1, C::TP, [](int i, int c) { return (long long)col_first<C>(i, c); }, root);
    return tab;
}

// The factors of a length are constants: built on the host by the first plan of that length (at most 1.2 MB over all seven lengths),
// copied to the device with each plan's other tables.
const std::vector<float4>* host_table(const m2_plan* pl) {
    if (pl->p < 2 || pl->p > 3) return nullptr;
    const std::vector<float4>* out = nullptr;
    dispatch(pl->N, [&](auto cfg) {
        static const std::vector<float4> tab = build_tab<decltype(cfg)>();
        out = &tab;
        return cudaSuccess;
    });
    return out;
}

// shared-memory limits of the kernels of this plan's length and type: once per device (bit d of the mask)
cudaError_t prepare(const m2_plan* pl) {
    static std::atomic<uint64_t> done[2][15];
    if (!covered(pl)) return cudaSuccess;
    std::atomic<uint64_t>& mask = done[pl->dtype == M2_BF16][log2_exact(pl->N)];
    const uint64_t bit = pl->device < 64 ? (uint64_t)1 << pl->device : 0;
    if (mask.load(std::memory_order_acquire) & bit) return cudaSuccess;
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        cudaError_t e = cudaSuccess;
        auto io = [&](auto z) {
            using IO = decltype(z);
            e = allow_smem(fft_conv_kernel<C, IO, false>, conv_smem<C>());
            if (e == cudaSuccess) e = allow_smem(fft_conv_kernel<C, IO, true>, conv_smem<C>());
        };
        if (pl->dtype == M2_BF16) io(__nv_bfloat16());
        else io(float());
        if (e == cudaSuccess) e = prepare_gradients(pl);
        if (e == cudaSuccess) mask.fetch_or(bit, std::memory_order_release);
        return e;
    });
}

cudaError_t conv(const m2_plan* pl, const void* x, const void* kf, void* y, int64_t B, int64_t H, int64_t n, bool causal, int kf_group,
                 cudaStream_t stream) {
    const long long npairs = (long long)((B + 1) / 2) * H;
    if (npairs == 0) return cudaSuccess;
    return dispatch(pl->N, [&](auto cfg) {
        using C = decltype(cfg);
        const unsigned grid = (unsigned)((npairs + C::ROWS - 1) / C::ROWS);
        auto go = [&](auto z, auto half) {
            using IO = decltype(z);
            return launch_early(fft_conv_kernel<C, IO, decltype(half)::v != 0>, grid, C::THREADS, conv_smem<C>(), stream, (const IO*)x,
                                (const float4*)kf, (IO*)y, (const float4*)pl->d_fft, (int)B, (int)H, (int)n, npairs, kf_group);
        };
        if (pl->dtype == M2_BF16) return causal ? go(__nv_bfloat16(), Ic<1>{}) : go(__nv_bfloat16(), Ic<0>{});
        return causal ? go(float(), Ic<1>{}) : go(float(), Ic<0>{});
    });
}

}  // namespace m2f
