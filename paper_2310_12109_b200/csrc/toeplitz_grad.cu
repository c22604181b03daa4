// Kernel gradient of short convolutions as products of segments on the tensor cores (bf16, N = 512):
//   dk[d] = sum over b, t of g[b][t] x[b][(t - d) mod N].
//
// With t = 128 p + t' and x cut into blocks of 64 positions, the products that share p, t' and the distance rho = 2 p - block are one matrix
// product over K = (p, b): D[t'][64 m + j'] = sum over p, b of g[b][128 p + t'] x[b][64 (2 p - top + m) + j'], and an element belongs to
// d = 64 top + t' - (64 m + j'): dk is the sum of D along its diagonals.  Both operands are taken as the TMA delivers them (blocks of
// [32 or 16 batch rows][64 positions], 128-byte swizzle, M/N-major: K runs over slots and rows); blocks before the row are zeros (causal); a
// circular row's first two blocks come a second time from L2, so that every run of four lies in consecutive slots.  n = 512: two accumulators of
// 256 columns (distances 0 .. 3 and 4 .. 7); causal n <= 256: one, the two halves of tensor memory taking channels in turn.
// Products of bf16 values are exact and their sums fp32: no operand and no partial sum is rounded to bf16, no partial sums go through memory and no
// inverse transform follows.  An accumulator is one chain over all batch rows, and the tensor core drops what lies below its last bit: the distance
// from 64 bits is 1.4e-7 for 32 rows of 512, 1.0e-6 for 256, 4.4e-6 for 1024 (fp32 transforms, the call without a workspace: 2.0e-7 to 2.9e-7).
//
// Diagonal sums: a warp reads its 32 rows x 128 columns as 8 x 8 blocks, each lane holding the same two places of every block
// (tcgen05.ld 16x256b), so the blocks along a diagonal are added without leaving the lane: 64 blocks become 19 bands, which 35 shuffles fold into
// 160 consecutive lags.  The warps' windows of lags are added through shared memory in a fixed order: results do not vary between calls.  Two
// sets of eight warps: circular, each has an accumulator of every channel; causal, they take the channels in turn.  A channel's windows are added
// after the next one's accumulator has been read, when every warp's have long arrived.
//
// Measured, one B200, us a launch, against bf16 transforms of both operands, partial spectra and an inverse transform (distance from 64 bits 3.0e-3):
// [32][768][512] circular 30.0 and 14.0, [8][768] 13.2 and 11.1, [8][4096] 34.5 and 38.8; causal [32][768][256] 29.1 and 7.3, [8][4096] 33.1
// and 23.  Up to 16 rows a channel costs the summing warps ~2400 cycles, whatever its rows (its 8 UMMAs take 1024): short batches of more than ~1500
// channels are where the transforms were faster.  With 32 rows the copies (72 KB a channel) and 16 UMMAs of 128 cycles come to as much.
// Sets that took whole channels in turn, each with both accumulators, a chain of two reads, two folds and an exchange: 15.5, 14.3, 52 us; the x row
// twice over (14 slots): 15.7 and 44 at [32][768] and [8][4096]; eight slots and UMMAs of 128 columns where a run wraps: 14.8 and 39.3.
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

constexpr int kSumWarps = 8, kSets = 2, kLoadWarp = kSets * kSumWarps, kIssueWarp = kLoadWarp + 1, kGradThreads = 32 * (kIssueWarp + 1);
constexpr int kBands = 19, kWindow = 8 * (kBands + 1);   // diagonals of 8 x 8 blocks in 32 rows x 128 columns; the lags they hold
constexpr int kRed = kSumWarps * kWindow * 4;            // one accumulator's windows of a set's warps

template <bool CIRC, int ROWS>   // circular n = 512, or causal n <= 256; batch rows per chunk
struct GCfg {
    static constexpr int SLOT = ROWS * 128;
    static constexpr int P = CIRC ? 4 : 2;                 // groups of 128 positions t
    static constexpr int GS = 2 * P, XS = CIRC ? 10 : 6;   // slots of g and x
    static constexpr int GROUPS = CIRC ? 2 : 1;            // accumulators per channel
    static constexpr int STAGE = (GS + XS) * SLOT;
    static constexpr int STAGES = CIRC ? (ROWS == 32 ? 2 : 5) : 4 * 32 / ROWS;
    static constexpr int OFF_RED = STAGES * STAGE;
    static constexpr int OFF_BAR = OFF_RED + 2 * kSets * kRed;   // two per set: a warp may be a channel ahead
    static constexpr int SMEM = OFF_BAR + 256;
};
static_assert(GCfg<true, 32>::SMEM <= 232448 && GCfg<false, 32>::SMEM <= 232448 && GCfg<true, 16>::SMEM <= 232448 && GCfg<false, 16>::SMEM <= 232448, "shared memory budget");

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

template <bool CIRC, int ROWS>
__global__ void __launch_bounds__(kGradThreads, 1)
    toeplitz_grad_kernel(const __grid_constant__ CUtensorMap mx, const __grid_constant__ CUtensorMap mg, float* __restrict__ dk, int H, int n,
                         int chunks, int32_t* __restrict__ status) {
    using C = GCfg<CIRC, ROWS>;
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t s0 = smem_u32(smem);
    const uint32_t bar_f = s0 + C::OFF_BAR, bar_e = bar_f + 8 * C::STAGES, bar_df = bar_e + 8 * C::STAGES, bar_de = bar_df + 16, bar_r = bar_de + 16,
                   s_tptr = bar_r + 8 * kSets;
    volatile uint32_t* tptr = reinterpret_cast<volatile uint32_t*>(smem + (s_tptr - s0));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + (s_tptr - s0) + 4);
    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(bar_f + 8 * s, 1);
            mbar_init(bar_e + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {   // an accumulator is one set's
            mbar_init(bar_df + 8 * a, 1);
            mbar_init(bar_de + 8 * a, kSumWarps);
            mbar_init(bar_r + 8 * a, CIRC ? kSets * kSumWarps : kSumWarps);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (!CIRC) {   // the blocks before a row are zero for good
        for (int i = tid; i < C::STAGES * 2 * (C::SLOT / 16); i += kGradThreads) {
            const int st = i / (2 * (C::SLOT / 16)), r = i % (2 * (C::SLOT / 16));
            *reinterpret_cast<uint4*>(smem + st * C::STAGE + C::GS * C::SLOT + r * 16) = make_uint4(0, 0, 0, 0);
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
                    const uint32_t ga = s0 + s * C::STAGE, xa = ga + C::GS * C::SLOT, bar = bar_f + 8 * s;
                    mbar_expect_tx(bar, (uint32_t)((C::GS + (CIRC ? C::XS : 4)) * C::SLOT));
                    for (int j = 0; j < C::GS; ++j) tma_load_4d(ga + j * C::SLOT, &mg, 64 * j, h, ch * ROWS, 0, bar);
                    if (CIRC) {
                        for (int j = 0; j < C::XS; ++j) tma_load_4d(xa + j * C::SLOT, &mx, 64 * ((j + 1) & 7), h, ch * ROWS, 0, bar);
                    } else {
                        for (int j = 0; j < 4; ++j) tma_load_4d(xa + (j + 2) * C::SLOT, &mx, 64 * j, h, ch * ROWS, 0, bar);
                    }
                }
            for (int i = v > C::STAGES ? v - C::STAGES : 0; i < v && ok; ++i) ok = mbar_wait(bar_e + 8 * (i % C::STAGES), (i / C::STAGES) & 1);
        }
    } else if (warp == kIssueWarp) {
        constexpr uint32_t idesc = instr_desc_bf16(128, 256, true, true);
        const uint64_t da0 = smem_desc_sw128(s0, C::SLOT, 1024), db0 = smem_desc_sw128(s0 + C::GS * C::SLOT, C::SLOT, 1024);
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
                        const uint64_t da = da0 + (uint32_t)(s * C::STAGE >> 4), db = db0 + (uint32_t)(s * C::STAGE >> 4);
#pragma unroll
                        for (int p = 0; p < C::P; ++p)
#pragma unroll
                            for (int ks = 0; ks < ROWS / 16; ++ks) {
                                const int sl = C::GROUPS == 2 ? (2 * p + 4 - 4 * gr) & 7 : 2 * p;   // the first of the four slots that meet segment p
                                umma_f16(tmem + a * 256, da + (uint32_t)((2 * p * C::SLOT + ks * 2048) >> 4), db + (uint32_t)((sl * C::SLOT + ks * 2048) >> 4), idesc,
                                         ch != 0 || p != 0 || ks != 0);
                            }
                        if (ch == chunks - 1) umma_commit(bar_df + 8 * a);
                        if (gr == C::GROUPS - 1) umma_commit(bar_e + 8 * s);
                    }
                    __syncwarp();
                }
            }
    } else {
        const int set = warp / kSumWarps, sw = warp % kSumWarps, q = warp & 3, hc = sw >> 2;   // rows 32 q .. of the set's accumulator, columns 128 hc ..
        const int r = lane >> 2, m = lane & 3, from1 = ((r + (m & 1 ? -2 : 2)) & 7) << 2 | (m ^ 1), from2 = (r ^ 4) << 2 | (m ^ 2);
        // circular: both sets take every channel, an accumulator each; causal: they take the channels in turn
        const int step = CIRC ? gridDim.x : kSets * gridDim.x;
        const uint32_t bar_set = bar_r + (CIRC ? 0 : 8 * set);
        float* const red = reinterpret_cast<float*>(smem + C::OFF_RED) + (CIRC ? 0 : 2 * set) * kSumWarps * kWindow;
        constexpr int kBuf = (CIRC ? kSets : 1) * kSumWarps * kWindow;   // the windows of a channel; two buffers
        // dk of the channel hp, the j-th of this warp.  The window of (set, q, hc) begins at lag 64 top + 32 q - 128 hc - 128, top = 3 and 7 (circular,
        // modulo 512), 2 (causal), and holds five times 32 lags: 32 lags lie in the windows q = c - 4 .. c of each hc, whose block c - q of 32 they
        // are; circular, c < 8 in one of the sets.
        auto finish = [&](int hp, int j) {
            bool done = mbar_wait(bar_set, j & 1);
            if (!__all_sync(0xffffffffu, done && *abort_flag == 0)) return false;
            const int d = 32 * (CIRC ? warp : sw) + lane;
            float sum = 0.f;
#pragma unroll
            for (int hz = 0; hz < 2; ++hz) {
                int c = (CIRC ? warp - 2 : sw) + 4 * hz;
                const int z = CIRC ? (c >> 3) & 1 : 0;
                if (CIRC) c &= 7;
                const float* w = red + (j & 1) * kBuf + (z * kSumWarps + 4 * hz) * kWindow + 32 * c + lane;
#pragma unroll
                for (int qz = 0; qz < 4; ++qz)
                    if (c - qz >= 0 && c - qz <= 4) sum += w[qz * (kWindow - 32)];
            }
            if (d < n) dk[(size_t)hp * n + d] = sum;
            return true;
        };
        int j = 0;
        for (int h = blockIdx.x + (CIRC ? 0 : set * gridDim.x); h < H; h += step, ++j) {
            ok = mbar_wait(bar_df + 8 * set, j & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            tc_fence_after();
            uint64_t band[kBands];   // block (R, k) of 8 x 8 adds to band R - k + 15
#pragma unroll
            for (int z = 0; z < kBands; ++z) band[z] = 0ull;
            const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + set * 256 + hc * 128;
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
                        uint64_t& b = band[R - (4 * c + k) + 15];
                        b = add2(b, pk2(v[R >> 1][4 * k + 2 * (R & 1)], v[R >> 1][4 * k + 2 * (R & 1) + 1]));
                    }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_de + 8 * set);
            if (j > 0) {   // the channel before: its windows have had this one's wait and loads to arrive in
                ok = finish(h - step, j - 1);
                if (!ok) break;
            }
            // lags 8 z + 0 .. 7 of the window: places with row - column = i of band z - 1 and i - 8 of band z; lane (r, m) gets lag 8 (4 y + m) + (r - 2 m mod 8).
            // (The buffer was read two channels ago; every warp has been through that when the barrier of the last one, just waited for, completed.)
            float* win = red + (j & 1) * kBuf + (CIRC ? warp : sw) * kWindow;
#pragma unroll
            for (int y = 0; y < 5; ++y) {
                float t[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int z = 4 * y + e;
                    float lox = 0.f, loy = 0.f, upx = 0.f, upy = 0.f;
                    if (z > 0) upk2(band[z - 1], lox, loy);
                    if (z < kBands) upk2(band[z], upx, upy);
                    const float v0 = r >= 2 * m ? lox : upx, v1 = r > 2 * m ? loy : upy;
                    t[e] = v0 + __shfl_sync(0xffffffffu, v1, lane + 4);   // (row r + 1, column 2 m + 1) joins (row r, column 2 m): i = r - 2 m
                }
                // the same i is two rows further down a column pair to the right, four rows two of them
                const float s01 = (m & 1 ? t[1] : t[0]) + __shfl_sync(0xffffffffu, m & 1 ? t[0] : t[1], from1);
                const float s23 = (m & 1 ? t[3] : t[2]) + __shfl_sync(0xffffffffu, m & 1 ? t[2] : t[3], from1);
                win[32 * y + 8 * m + ((r - 2 * m) & 7)] = (m & 2 ? s23 : s01) + __shfl_sync(0xffffffffu, m & 2 ? s01 : s23, from2);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_set);
        }
        if (ok && j > 0) ok = finish(blockIdx.x + (CIRC ? 0 : set * gridDim.x) + (j - 1) * step, j - 1);
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
    // Up to 16 batch rows: chunks of 16, half the copies and UMMAs (K = 16 is the least): [8][4096][512] circular 52 -> 47 us with the kernel as it was
    const int rows = B <= 16 ? 16 : 32;
    auto kern = causal ? (rows == 16 ? toeplitz_grad_kernel<false, 16> : toeplitz_grad_kernel<false, 32>)
                       : (rows == 16 ? toeplitz_grad_kernel<true, 16> : toeplitz_grad_kernel<true, 32>);
    const int smem = causal ? (rows == 16 ? GCfg<false, 16>::SMEM : GCfg<false, 32>::SMEM) : (rows == 16 ? GCfg<true, 16>::SMEM : GCfg<true, 32>::SMEM);
    alignas(64) CUtensorMap m[2];
    const void* const src[2] = {x, g};
    for (int i = 0; i < 2; ++i) {   // box: 64 positions of a chunk's batch rows
        const cuuint64_t gdim[4] = {(cuuint64_t)n, (cuuint64_t)H, (cuuint64_t)B, 1};
        const cuuint64_t gstr[3] = {(cuuint64_t)n * 2, (cuuint64_t)H * n * 2, (cuuint64_t)B * H * n * 2};
        const cuuint32_t box[4] = {64, 1, (cuuint32_t)rows, 1};
        if (!tma_host::encode_sw128_bf16(&m[i], src[i], 4, gdim, gstr, box)) return M2_ERR_UNSUPPORTED;
    }
    static std::atomic<uint32_t> done[64];   // bit per kernel
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return M2_ERR_CUDA;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool known = dev >= 0 && dev < 64;
    const uint32_t bit = 1u << ((causal ? 2 : 0) + (rows == 16 ? 1 : 0));
    if (!known || !(done[dev].load(std::memory_order_acquire) & bit)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return M2_ERR_CUDA;
        if (known) done[dev].fetch_or(bit, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(H < sms ? H : sms));
    cfg.blockDim = dim3(kGradThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int chunks = (int)((B + rows - 1) / rows);
    if (cudaLaunchKernelEx(&cfg, kern, m[0], m[1], dk, (int)H, (int)n, chunks, pl->d_status) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->last_kernel = "conv_wgrad_toeplitz";
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2t
