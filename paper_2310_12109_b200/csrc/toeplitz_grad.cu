// Kernel gradient of short convolutions as products of segments on the tensor cores (bf16, N = 512):
//   dk[d] = sum over b, t of g[b][t] x[b][(t - d) mod N].
//
// With t = 128 p + t' and x cut into blocks of 64 positions, the products that share p, t' and the distance rho = 2 p - block are one matrix
// product over K = (p, b): D[t'][64 m + j'] = sum over p, b of g[b][128 p + t'] x[b][64 (2 p - top + m) + j'], and an element belongs to
// d = 64 top + t' - (64 m + j'): dk is the sum of D along its diagonals.  Both operands are taken as the TMA delivers them (blocks of
// [32 batch rows][64 positions], 128-byte swizzle, M/N-major: K runs over slots and rows); blocks before the row are zeros (causal) or come a
// second time from L2 (circular).  n = 512: two accumulators of 256 columns (distances 0 .. 3 and 4 .. 7); causal n <= 256: one, the two
// halves of tensor memory taking channels in turn.
// Products of bf16 values are exact and everything after them is fp32: nothing is rounded between the inputs and dk, no partial sums go
// through memory and no inverse transform follows.
//
// Diagonal sums: a warp reads its 32 rows x 128 columns as 8 x 8 blocks, each lane holding the same two places of every block
// (tcgen05.ld 16x256b), so the blocks along a diagonal are added without leaving the lane: 64 blocks become 19 bands, which 55 shuffles fold into
// 160 consecutive lags.  The warps' windows of lags are added through shared memory in a fixed order: results do not vary between calls.  Two
// sets of eight warps take the channels in turn: the chain of a channel (waits, two accumulators, one exchange) is longer than its products.
//
// Measured, one B200 (call with its host work): [32][768][512] circular 31.6 -> 16.5 us, [32][768][256] causal 30.4 -> 11.4, [256][768][256] 181 ->
// 37.7, against bf16 transforms of both operands, partial spectra and an inverse transform; distance from 64 bits 3.0e-3 -> 1.4e-7.  Bound by a
// block's copies (88 KB a channel of 32 rows, of which 24 from L2) and its 16 UMMAs of 128 cycles, both ~2000 cycles of the ~2600 it takes; short
// calls by launch and host.  With one shuffle per element instead of the bands the same took 22.5 us, with bands whose cross-warp sum waited
// twice per accumulator 30.
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>

#include "m2_plan.h"
#include "ptx_sm100.cuh"
#include "tma_host.h"
#include "toeplitz_mma.h"

namespace m2t {

using namespace sm100;

namespace {

constexpr int kGRows = 32, kGSlot = kGRows * 128;
constexpr int kSumWarps = 8, kSets = 2, kLoadWarp = kSets * kSumWarps, kIssueWarp = kLoadWarp + 1, kGradThreads = 32 * (kIssueWarp + 1);
constexpr int kBands = 19, kWindow = 8 * (kBands + 1);   // diagonals of 8 x 8 blocks in 32 rows x 128 columns; the lags they hold
constexpr int kRed = kSumWarps * kWindow * 4;            // one accumulator's windows of a set's warps

template <bool CIRC>   // circular n = 512, or causal n <= 256
struct GCfg {
    static constexpr int P = CIRC ? 4 : 2;                 // groups of 128 positions t
    static constexpr int GS = 2 * P, XS = CIRC ? 14 : 6;   // slots of g and x
    static constexpr int GROUPS = CIRC ? 2 : 1;            // accumulators per channel
    static constexpr int STAGE = (GS + XS) * kGSlot;
    static constexpr int STAGES = CIRC ? 2 : 4;
    static constexpr int OFF_RED = STAGES * STAGE;
    static constexpr int OFF_BAR = OFF_RED + 2 * kSets * GROUPS * kRed;   // two per set: a warp may be a channel ahead
    static constexpr int SMEM = OFF_BAR + 256;
};
static_assert(GCfg<true>::SMEM <= 232448 && GCfg<false>::SMEM <= 232448, "shared memory budget");

// 16 rows x 32 columns: registers 4 n .. 4 n + 3 are (row, column) (l / 4, 8 n + 2 (l % 4)), the next column, and both again 8 rows below
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
                   "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

template <bool CIRC>
__global__ void __launch_bounds__(kGradThreads, 1)
    toeplitz_grad_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mg, float* __restrict__ dk, int H, int n,
                         int chunks, int32_t* __restrict__ status) {
    using C = GCfg<CIRC>;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t s0 = smem_u32(smem);
    const uint32_t bar_f = s0 + C::OFF_BAR, bar_e = bar_f + 8 * C::STAGES, bar_df = bar_e + 8 * C::STAGES, bar_de = bar_df + 8 * kSets * C::GROUPS, bar_r = bar_de + 16,
                   s_tptr = bar_r + 8 * kSets;
    volatile uint32_t* tptr = reinterpret_cast<volatile uint32_t*>(smem + (s_tptr - s0));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + (s_tptr - s0) + 4);
    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(bar_f + 8 * s, 1);
            mbar_init(bar_e + 8 * s, 1);
        }
        for (int z = 0; z < kSets * C::GROUPS; ++z) mbar_init(bar_df + 8 * z, 1);   // per set: neither waits on a phase of the other's
        for (int a = 0; a < 2; ++a) mbar_init(bar_de + 8 * a, kSumWarps);
        for (int z = 0; z < kSets; ++z) mbar_init(bar_r + 8 * z, kSumWarps);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (!CIRC) {   // the blocks before a row are zero for good
        for (int i = tid; i < C::STAGES * 2 * (kGSlot / 16); i += kGradThreads) {
            const int st = i / (2 * (kGSlot / 16)), r = i % (2 * (kGSlot / 16));
            *reinterpret_cast<uint4*>(smem + st * C::STAGE + C::GS * kGSlot + r * 16) = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async();
    }
    if (warp == kIssueWarp) tmem_alloc(s_tptr, 512);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *tptr;
    bool ok = true;

    if (warp == kLoadWarp) {
        if (lane == 0) {
            int v = 0;
            for (int h = blockIdx.x; h < H && ok; h += gridDim.x)
                for (int ch = 0; ch < chunks; ++ch, ++v) {
                    const int s = v % C::STAGES;
                    if (v >= C::STAGES) ok = mbar_wait(bar_e + 8 * s, (v / C::STAGES - 1) & 1);
                    if (!ok || *abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t ga = s0 + s * C::STAGE, xa = ga + C::GS * kGSlot, bar = bar_f + 8 * s;
                    mbar_expect_tx(bar, (uint32_t)((C::GS + (CIRC ? C::XS : 4)) * kGSlot));
                    for (int j = 0; j < C::GS; ++j) tma_load_4d(ga + j * kGSlot, &mg, 64 * j, h, ch * kGRows, 0, bar);
                    if (CIRC) {
                        for (int j = 0; j < C::XS; ++j) tma_load_4d(xa + j * kGSlot, &mx, 64 * ((j + 1) & 7), h, ch * kGRows, 0, bar);
                    } else {
                        for (int j = 0; j < 4; ++j) tma_load_4d(xa + (j + 2) * kGSlot, &mx, 64 * j, h, ch * kGRows, 0, bar);
                    }
                }
            for (int i = v > C::STAGES ? v - C::STAGES : 0; i < v && ok; ++i) ok = mbar_wait(bar_e + 8 * (i % C::STAGES), (i / C::STAGES) & 1);
        }
    } else if (warp == kIssueWarp) {
        constexpr uint32_t idesc = instr_desc_bf16(128, 256, true, true);
        const uint64_t da0 = smem_desc_sw128(s0, kGSlot, 1024), db0 = smem_desc_sw128(s0 + C::GS * kGSlot, kGSlot, 1024);
        int v = 0, it = 0;
        for (int h = blockIdx.x; h < H && ok; h += gridDim.x, ++it)
            for (int ch = 0; ch < chunks && ok; ++ch, ++v) {
                const int s = v % C::STAGES;
                ok = mbar_wait(bar_f + 8 * s, (v / C::STAGES) & 1);
                ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
#pragma unroll
                for (int gr = 0; gr < C::GROUPS; ++gr) {
                    const int use = C::GROUPS == 2 ? it : it >> 1, a = C::GROUPS == 2 ? gr : it & 1;   // the accumulator and how often it was used before
                    if (ok && ch == 0 && use > 0) ok = mbar_wait(bar_de + 8 * a, (use - 1) & 1);
                    ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint64_t da = da0 + (uint32_t)(s * C::STAGE >> 4), db = db0 + (uint32_t)((s * C::STAGE + (C::GROUPS == 2 ? 4 - 4 * gr : 0) * kGSlot) >> 4);
#pragma unroll
                        for (int p = 0; p < C::P; ++p)
#pragma unroll
                            for (int ks = 0; ks < 2; ++ks)
                                umma_f16(tmem + a * 256, da + (uint32_t)((2 * p * kGSlot + ks * 2048) >> 4), db + (uint32_t)((2 * p * kGSlot + ks * 2048) >> 4), idesc,
                                         ch != 0 || p != 0 || ks != 0);
                        if (ch == chunks - 1) umma_commit(bar_df + 8 * (it % kSets * C::GROUPS + gr));
                        if (gr == C::GROUPS - 1) umma_commit(bar_e + 8 * s);
                    }
                    __syncwarp();
                }
            }
    } else {
        const int set = warp / kSumWarps, sw = warp % kSumWarps, q = warp & 3, hc = sw >> 2;   // rows 32 q .. of the accumulators, columns 128 hc ..
        const int r = lane >> 2, m = lane & 3;
        int it = set;
        for (int h = blockIdx.x + set * gridDim.x; h < H && ok; h += kSets * gridDim.x, it += kSets) {
            float* red = reinterpret_cast<float*>(smem + C::OFF_RED) + (set * 2 + ((it / kSets) & 1)) * C::GROUPS * kSumWarps * kWindow;
#pragma unroll 1
            for (int gr = 0; gr < C::GROUPS; ++gr) {
                const int a = C::GROUPS == 2 ? gr : it & 1;
                ok = mbar_wait(bar_df + 8 * (set * C::GROUPS + gr), (it / kSets) & 1);
                ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
                if (!ok) break;
                tc_fence_after();
                float2 band[kBands];   // block (R, k) of 8 x 8 adds to band R - k + 15
#pragma unroll
                for (int z = 0; z < kBands; ++z) band[z] = make_float2(0.f, 0.f);
                const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + a * 256 + hc * 128;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float v[2][16];
                    tmem_ld_16x32(tcol + 32 * c, v[0]);
                    tmem_ld_16x32(tcol + (16u << 16) + 32 * c, v[1]);
                    tmem_ld_wait();
#pragma unroll
                    for (int z = 0; z < 4; ++z) tmem_ld_fence8(&v[0][0] + 8 * z);
#pragma unroll
                    for (int R = 0; R < 4; ++R)
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            float2& b = band[R - (4 * c + k) + 15];
                            b.x += v[R >> 1][4 * k + 2 * (R & 1)];
                            b.y += v[R >> 1][4 * k + 2 * (R & 1) + 1];
                        }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_de + 8 * a);
                // lags 8 z + 0 .. 7 of the window: places with row - column = i of band z - 1 and i - 8 of band z; lane (r, m) gets lag 8 (4 j + m) + r
#pragma unroll
                for (int j = 0; j < 5; ++j) {
                    float t[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int z = 4 * j + e;
                        const float2 lo = z > 0 ? band[z - 1] : make_float2(0.f, 0.f), up = z < kBands ? band[z] : make_float2(0.f, 0.f);
                        const float v0 = r >= 2 * m ? lo.x : up.x, v1 = r > 2 * m ? lo.y : up.y;
                        t[e] = v0 + __shfl_sync(0xffffffffu, v1, lane + 4);   // (row r + 1, column 2 m + 1) joins (row r, column 2 m)
                        t[e] = __shfl_sync(0xffffffffu, t[e], lane + 8 * m);   // i = r - 2 m: the four columns' rows side by side
                    }
                    const float s01 = (m & 1 ? t[1] : t[0]) + __shfl_xor_sync(0xffffffffu, m & 1 ? t[0] : t[1], 1);
                    const float s23 = (m & 1 ? t[3] : t[2]) + __shfl_xor_sync(0xffffffffu, m & 1 ? t[2] : t[3], 1);
                    red[(gr * kSumWarps + sw) * kWindow + 32 * j + 8 * m + r] = (m & 2 ? s23 : s01) + __shfl_xor_sync(0xffffffffu, m & 2 ? s01 : s23, 2);
                }
            }
            if (!ok) break;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_r + 8 * set);
            ok = mbar_wait(bar_r + 8 * set, (it / kSets) & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            // the window of (gr, q, hc) begins at lag 64 top + 32 q - 128 hc - 128, top = 3 and 7 (circular, modulo 512), 2 (causal).  (The set's
            // next channel goes to the other buffer; this one is written again when every warp of the set has passed here.)
#pragma unroll
            for (int z = 0; z < (CIRC ? 2 : 1); ++z) {
                const int d = 32 * sw + lane + 256 * z;
                float sum = 0.f;
#pragma unroll
                for (int gr = 0; gr < C::GROUPS; ++gr)
#pragma unroll
                    for (int w = 0; w < kSumWarps; ++w) {
                        int o = d - 64 * (CIRC ? 3 + 4 * gr : 2) - 32 * (w & 3) + 128 * (w >> 2) + 128;
                        if (CIRC) o &= 511;
                        if (o >= 0 && o < kWindow) sum += red[(gr * kSumWarps + w) * kWindow + o];
                    }
                if (d < n) dk[(size_t)h * n + d] = sum;
            }
        }
    }
    if (!ok && lane == 0) {
        *abort_flag = 1;
        atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // copies issued before the wait ran out have landed by then
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kIssueWarp) tmem_dealloc(tmem, 512);
}

}  // namespace

// A channel's batch rows are one block's work: few channels with many rows stay with the kernel whose units are 8 rows ([1024][4][512] 20.4 us
// there, [256][4] 14.4 there and 14.0 here, [256][64] 26.7 and 15.6).
bool grad_covers(const m2_plan* pl, int64_t B, int64_t H, int64_t n, bool causal) {
    if (pl->dtype != M2_BF16 || pl->N != 512 || (causal ? n % 16 != 0 || n > 256 : n != 512)) return false;
    return B <= 256 || H >= 64;
}

int32_t conv_grad(const m2_plan* pl, const void* x, const void* g, float* dk, int64_t B, int64_t H, int64_t n, bool causal, cudaStream_t stream) {
    if (!grad_covers(pl, B, H, n, causal) || B > 0x7fffffffLL || H > 0x7fffffffLL) return M2_ERR_UNSUPPORTED;
    alignas(64) CUtensorMap m[2];
    const void* const src[2] = {x, g};
    for (int i = 0; i < 2; ++i) {   // box: 64 positions of 32 batch rows
        const cuuint64_t gdim[4] = {(cuuint64_t)n, (cuuint64_t)H, (cuuint64_t)B, 1};
        const cuuint64_t gstr[3] = {(cuuint64_t)n * 2, (cuuint64_t)H * n * 2, (cuuint64_t)B * H * n * 2};
        const cuuint32_t box[4] = {64, 1, (cuuint32_t)kGRows, 1};
        if (!tma_host::encode_sw128_bf16(&m[i], src[i], 4, gdim, gstr, box)) return M2_ERR_UNSUPPORTED;
    }
    static std::atomic<bool> done[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return M2_ERR_CUDA;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool known = dev >= 0 && dev < 64;
    if (!known || !done[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(toeplitz_grad_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<true>::SMEM) != cudaSuccess ||
            cudaFuncSetAttribute(toeplitz_grad_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, GCfg<false>::SMEM) != cudaSuccess)
            return M2_ERR_CUDA;
        if (known) done[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(H < sms ? H : sms));
    cfg.blockDim = dim3(kGradThreads);
    cfg.dynamicSmemBytes = causal ? GCfg<false>::SMEM : GCfg<true>::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int chunks = (int)((B + kGRows - 1) / kGRows);
    if (cudaLaunchKernelEx(&cfg, causal ? toeplitz_grad_kernel<false> : toeplitz_grad_kernel<true>, m[0], m[1], dk, (int)H, (int)n, chunks, pl->d_status) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2t
