// Short causal convolutions (bf16, 160 < n <= 256) as Toeplitz products on the fifth-generation tensor cores:
//   y[b][t] = sum_j k[t - j] x[b][j] per channel.
//
// A channel's T(k) is n x n, but only its diagonals differ.  Rows are cut into four segments of S = 64 positions and the UMMA's M index is
// (segment p, batch row b), 4 x 32 = 128; shifting x by a segment per p makes one T of S columns serve all four:
//   y[b][p S + t'] = sum_j'' x[b][j'' + p S] k[t' - j''],      -3 S <= j'' < S  (further up where k has lags below zero).
//   * A = x as the TMA delivers it: slots of [32 batch rows][64 positions] with the 128-byte swizzle, segment after segment; "segment + 1" is
//     the next slot, so the shift by p S is the uniform stride between groups of 8 rows.  Segments outside a row are slots of zeros.
//   * B = T(k) from an image of its DIFFERENT 8 x 8 core matrices, one per diagonal: core matrix (I, J) lies at base + (I' + J) 256 with
//     I' = S / 8 - 1 - I, i.e. the descriptor's strides walk the diagonals (output groups come out in reverse order, which the epilogue
//     undoes).  10 KB stand for 2 x 32 KB of operand.
//   * The kernel is fp32: its values are split into two bf16 parts and both are multiplied; the parts' core matrices alternate, so N = 2 S
//     columns hold both products and the epilogue adds them in fp32.
// Nothing is rounded between x and the one rounding of y.
//
// An item is one channel and 32 batch rows; persistent blocks, one per SM, whose roles meet through mbarriers: a TMA warp, four warps that
// build the images, an issuing warp, eight epilogue warps.
//
// Measured, one B200: [32][768][256] 15.7 -> 11.9 us against the mma.sync kernel, the three convolutions of the Hyena layer at that size in one
// launch 40 -> 28 us (cold).  Bound by shared memory: an item's 16 UMMAs read 8 KB each for 64 cycles of tensor work, 1900 of the ~2100 cycles an
// item takes; the images, the copies in and the staging take the rest of its bandwidth.  Circular rows of 512 the same way (S = 128, N = 256
// columns: 32 UMMAs of 142 cycles per item) took 23.1 us against 19.8 for the row-pair transforms: 25.8 GFLOP where those need a fraction of it.
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

constexpr int S = 64;         // positions per segment
constexpr int kRowsPerItem = 32, kSlot = kRowsPerItem * 128;   // a slot: 32 batch rows x 64 positions
constexpr int kEpiWarps = 8, kBuildWarps = 4, kTmaWarp = 12, kMmaWarp = 13;
constexpr int kUmmaThreads = 32 * 14;
constexpr int kKBuf = 2048;   // a kernel row: up to 512 fp32 values
constexpr int kKRows = 2;     // ... of which this many are on their way
constexpr int kImages = 2;

constexpr int kOwnDiag = 3 * S / 8, kDiags = 5 * S / 8 - 1, kAllDiags = 8 * S / 8 - 1;   // core matrices of one part: the first of a segment with itself; lags above -64; all
constexpr int kAcc = 512 / (2 * S);                                // accumulators of 2 S columns

constexpr int kSlots = 10, kStages = 3;                            // segments -3 .. 3, and up to 6 for lags below zero
constexpr int kXBuf = kSlots * kSlot, kBBuf = (kAllDiags * 256 + 1023) / 1024 * 1024;
constexpr int kOffB = kStages * kXBuf;
constexpr int kOffStg = kOffB + kImages * kBBuf;                   // 4 KB per epilogue warp: the image of a [32][64] output box
constexpr int kOffK = kOffStg + kEpiWarps * kSlot;
constexpr int kOffBar = kOffK + kKRows * kKBuf;
constexpr int kUmmaSmem = kOffBar + 256;
static_assert(kUmmaSmem <= 232448, "shared memory budget");

struct UmmaArgs {
    CUtensorMap x[3], y[3];
    const float* kt[3];
    int H, n, N, kf_group;
    int per_set, items;    // items in the order set, batch chunk, channel
};

__device__ __forceinline__ uint32_t pack_bf2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_f(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__global__ void __launch_bounds__(kUmmaThreads, 1) toeplitz_umma_kernel(const __grid_constant__ UmmaArgs P, int32_t* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t s0 = smem_u32(smem);
    const uint32_t bar_xf = s0 + kOffBar, bar_xe = bar_xf + 8 * kStages, bar_kf = bar_xe + 8 * kStages, bar_ke = bar_kf + 8 * kKRows,
                   bar_bf = bar_ke + 8 * kKRows, bar_be = bar_bf + 8 * kImages, bar_df = bar_be + 8 * kImages, bar_de = bar_df + 8 * kAcc, s_tptr = bar_de + 8 * kAcc;
    static_assert(8 * (2 * kStages + 2 * kKRows + 2 * kImages + 2 * kAcc) + 8 + 4 * kImages <= 256, "barrier area");
    volatile uint32_t* tptr = reinterpret_cast<volatile uint32_t*>(smem + (s_tptr - s0));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + (s_tptr - s0) + 4);
    volatile uint32_t* flags = reinterpret_cast<volatile uint32_t*>(smem + (s_tptr - s0) + 8);   // [image]: lags above / below zero
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(bar_xf + 8 * s, 1);
            mbar_init(bar_xe + 8 * s, 1);
        }
        for (int s = 0; s < kKRows; ++s) {
            mbar_init(bar_kf + 8 * s, 1);
            mbar_init(bar_ke + 8 * s, kBuildWarps);
        }
        for (int s = 0; s < kImages; ++s) {
            mbar_init(bar_bf + 8 * s, kBuildWarps);
            mbar_init(bar_be + 8 * s, 1);
        }
        for (int s = 0; s < kAcc; ++s) {
            mbar_init(bar_df + 8 * s, 1);
            mbar_init(bar_de + 8 * s, kEpiWarps / 2);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    // the segments outside a row are zero for good
    for (int i = tid; i < kStages * 6 * (kSlot / 16); i += kUmmaThreads) {
        const int st = i / (6 * (kSlot / 16)), r = i % (6 * (kSlot / 16)), sl = r / (kSlot / 16);
        *reinterpret_cast<uint4*>(smem + st * kXBuf + (sl < 3 ? sl : sl + 4) * kSlot + (r % (kSlot / 16)) * 16) = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async();
    if (warp == kMmaWarp) tmem_alloc(s_tptr, 512);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the operands may have been written by the kernel before this one
    const uint32_t tmem = *tptr;
    bool ok = true;

    const int count = (P.items - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    auto item_of = [&](int i) { return i * (int)gridDim.x + (int)blockIdx.x; };

    if (warp == kTmaWarp) {
        if (lane == 0) {
            for (int i = 0; i < count && ok; ++i) {
                const int it = item_of(i), set = it / P.per_set, r = it - set * P.per_set, ch = r / P.H, h = r - ch * P.H;
                const int kb = i % kKRows, s = i % kStages;
                if (i >= kKRows) ok = mbar_wait(bar_ke + 8 * kb, (i / kKRows - 1) & 1);
                if (!ok || *abort_flag) {
                    ok = false;
                    break;
                }
                mbar_expect_tx(bar_kf + 8 * kb, (uint32_t)P.N * 4);
                bulk_load(s0 + kOffK + kb * kKBuf, P.kt[set] + (size_t)(h / P.kf_group) * P.N, (uint32_t)P.N * 4, bar_kf + 8 * kb);
                if (i >= kStages) ok = mbar_wait(bar_xe + 8 * s, (i / kStages - 1) & 1);
                if (!ok || *abort_flag) {
                    ok = false;
                    break;
                }
                const uint32_t xa = s0 + s * kXBuf;
                mbar_expect_tx(bar_xf + 8 * s, 4 * kSlot);
                for (int sg = 0; sg < 4; ++sg) tma_load_4d(xa + (sg + 3) * kSlot, &P.x[set], sg * S, h, ch * kRowsPerItem, 0, bar_xf + 8 * s);
            }
            for (int i = count > kStages ? count - kStages : 0; i < count && ok; ++i)   // stay until the last commits have arrived
                ok = mbar_wait(bar_xe + 8 * (i % kStages), (i / kStages) & 1);
        }
    } else if (warp == kMmaWarp) {
        constexpr uint32_t idesc = instr_desc_bf16(128, 2 * S, false, false);
        const uint64_t da0 = smem_desc_sw128(s0, 16, 1024), db0 = smem_desc(s0 + kOffB, 256, 128);
        bool b_in = false, x_in = false, d_out = true;   // what the next item waits for is known to have happened
        for (int i = 0; i < count && ok; ++i) {
            const int s = i % kStages, b = i % kImages, a = i % kAcc;
            if (!b_in) ok = mbar_wait(bar_bf + 8 * b, (i / kImages) & 1);
            if (ok && !x_in) ok = mbar_wait(bar_xf + 8 * s, (i / kStages) & 1);
            if (ok && !d_out) ok = mbar_wait(bar_de + 8 * a, (i / kAcc - 1) & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            tc_fence_after();
            const uint32_t f = flags[b];
            const int u0 = f & 1 ? 0 : 3, u1 = f & 2 ? 6 : 3;   // a side without a non-zero value is not walked
            const uint32_t d = tmem + a * 2 * S;
            const uint64_t da = da0 + (uint32_t)(s * kXBuf >> 4), db = db0 + (uint32_t)(b * kBBuf >> 4);
            auto segment = [&](int u) {
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    umma_f16(d, da + (uint32_t)((u * kSlot + ks * 32) >> 4), db + (uint32_t)((u * (S / 8) + ks * 2) * 256 >> 4), idesc, u != u0 || ks != 0);
            };
            if (elect_one())
                for (int u = u0; u < u1; ++u) segment(u);
            __syncwarp();
            // a wait takes ~150 cycles even where nothing is left to wait for: looked at while the tensor core has work
            if (i + 1 < count) {
                b_in = mbar_test(bar_bf + 8 * ((i + 1) % kImages), ((i + 1) / kImages) & 1);
                x_in = mbar_test(bar_xf + 8 * ((i + 1) % kStages), ((i + 1) / kStages) & 1);
                d_out = i + 1 < kAcc || mbar_test(bar_de + 8 * ((i + 1) % kAcc), ((i + 1) / kAcc - 1) & 1);
            }
            if (elect_one()) {
                segment(u1);
                umma_commit(bar_df + 8 * a);
                umma_commit(bar_xe + 8 * s);
                umma_commit(bar_be + 8 * b);
            }
            __syncwarp();
        }
    } else if (warp >= kEpiWarps) {
        const int bt = tid - 32 * kEpiWarps;
        for (int i = 0; i < count && ok; ++i) {
            const int kb = i % kKRows, b = i % kImages;
            ok = mbar_wait(bar_kf + 8 * kb, (i / kKRows) & 1);
            if (ok && i >= kImages) ok = mbar_wait(bar_be + 8 * b, (i / kImages - 1) & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            const float* k = reinterpret_cast<const float*>(smem + kOffK + kb * kKBuf);
            unsigned char* img = smem + kOffB + b * kBBuf;
            // lags that no pair of positions has are zero, whatever the spectrum's kernel holds there
            auto value = [&](int lag) { return lag >= P.n || lag <= -P.n ? 0.f : k[lag & (P.N - 1)]; };
            auto window = [&](int w) {   // row w & 7 of diagonal w >> 3: lags lag, lag - 1, .. lag - 7
                const int lag = 4 * S - 8 - 8 * (w >> 3) + (w & 7);
                uint32_t hi[4], lo[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const float v0 = value(lag - 2 * c), v1 = value(lag - 2 * c - 1);
                    hi[c] = pack_bf2(v0, v1);
                    lo[c] = pack_bf2(v0 - lo_f(hi[c]), v1 - hi_f(hi[c]));
                }
                uint4* dst = reinterpret_cast<uint4*>(img + (w >> 3) * 256 + (w & 7) * 16);
                dst[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                dst[8] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
            };
            bool later = false, earlier = false;   // (every building warp looks at all lags: they need not meet)
#pragma unroll
            for (int u = 1 + lane; u < 256; u += 32) {
                later = later || value(u) != 0.f;
                earlier = earlier || value(-u) != 0.f;
            }
            later = __any_sync(0xffffffffu, later);
            earlier = __any_sync(0xffffffffu, earlier);
            if (bt == 0) flags[b] = (later ? 1u : 0u) | (earlier ? 2u : 0u);
            // the diagonals that the walked segments reach
            for (int w = (later ? 0 : 8 * kOwnDiag) + bt; w < 8 * (earlier ? kAllDiags : kDiags); w += 32 * kBuildWarps) window(w);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_ke + 8 * kb);
                mbar_arrive(bar_bf + 8 * b);
            }
        }
        for (int i = count > kImages ? count - kImages : 0; i < count && ok; ++i) ok = mbar_wait(bar_be + 8 * (i % kImages), (i / kImages) & 1);
    } else {
        // epilogue: lane = batch row, warp & 3 = segment; the two sets of four warps take the items in turn
        const int q = warp & 3, sw = lane & 7;
        unsigned char* stg = smem + kOffStg + warp * kSlot + lane * 128;
        for (int i = warp >> 2; i < count && ok; i += 2) {
            const int it = item_of(i), set = it / P.per_set, r = it - set * P.per_set, ch = r / P.H, h = r - ch * P.H;
            const int a = i % kAcc;
            ok = mbar_wait(bar_df + 8 * a, (i / kAcc) & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            tc_fence_after();
            if (lane == 0) tma_store_wait_read0();   // the previous store has read the staging area
            __syncwarp();
            const uint32_t tcol = tmem + ((uint32_t)(q * 32) << 16) + a * 2 * S;
#pragma unroll
            for (int c2 = 0; c2 < 4; ++c2) {   // positions 16 c2 .. 16 c2 + 15: column groups 7 - 2 c2 and 6 - 2 c2
                float v[32];
                tmem_ld8(tcol + 16 * (7 - 2 * c2), v);
                tmem_ld8(tcol + 16 * (7 - 2 * c2) + 8, v + 8);
                tmem_ld8(tcol + 16 * (6 - 2 * c2), v + 16);
                tmem_ld8(tcol + 16 * (6 - 2 * c2) + 8, v + 24);
                tmem_ld_wait();
#pragma unroll
                for (int z = 0; z < 4; ++z) tmem_ld_fence8(v + 8 * z);
#pragma unroll
                for (int z = 0; z < 2; ++z) {
                    uint32_t o[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) o[t] = pack_bf2(v[16 * z + 2 * t] + v[16 * z + 8 + 2 * t], v[16 * z + 2 * t + 1] + v[16 * z + 9 + 2 * t]);
                    *reinterpret_cast<uint4*>(stg + (((2 * c2 + z) ^ sw) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar_de + 8 * a);
                if (q * S < P.n) {   // (rows past B and positions past n are clipped by the tensor map)
                    tma_store_4d(&P.y[set], s0 + kOffStg + warp * kSlot, q * S, h, ch * kRowsPerItem, 0);
                    tma_store_commit();
                }
            }
        }
        if (lane == 0) tma_store_wait_read0();   // the staging area dies with the block
    }
    if (!ok && lane == 0) {
        *abort_flag = 1;
        atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // copies issued before the wait ran out have landed by then
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

// rows [B][H][n] as a tensor; box: 64 positions of 32 batch rows, 128-byte swizzle
bool map_rows(CUtensorMap* m, const void* p, int64_t B, int64_t H, int64_t n) {
    const cuuint64_t gdim[4] = {(cuuint64_t)n, (cuuint64_t)H, (cuuint64_t)B, 1};
    const cuuint64_t gstr[3] = {(cuuint64_t)n * 2, (cuuint64_t)H * n * 2, (cuuint64_t)B * H * n * 2};
    const cuuint32_t box[4] = {64, 1, (cuuint32_t)kRowsPerItem, 1};
    return tma_host::encode_sw128_bf16(m, p, 4, gdim, gstr, box);
}

}  // namespace

// With the machine full an item takes 8.9 ns here, whatever n and the rows it holds; the mma.sync kernel's items of 32 rows take 12.7 (n =
// 256), 12.0 (200), 10.9 (192) and 8.7 ns (136), its items of 16 rows half of that.  One set, us, there and here: [32][768][256] 14.4 and 11.5,
// [33][768][216] 21.5 and 17.7, [32][768][192] 11.9 and 11.4, [16][768][256] 9.6 and 11.5.  This kernel starts 1.5 to 2 us later (set-up, tensor maps), and the
// other takes up to three items per SM, 444 in all, in one round; what its fourth to sixth cost grows with n.  Items, there and here, n = 256:
// [300] 7.5 and 7.3, [444] 7.6 and 8.2, [445] 9.5 and 8.6; 224: [444] 7.0 and 8.2, [445] 8.6 both, [520] 9.6 and 9.0; 192: [296] 5.0 and 6.9, [444] 6.4 and 8.1,
// [520] 8.8 and 8.9, [592] 10.8 and 9.4.  Shorter rows: two rounds of the other's, [888] 11.6 and 12.1, [1500] 19.8 and 17.7 (n = 168 .. 184); down to 160, where
// an item costs the same in both ([48][2400] 45.7 and 45.5).
bool umma_pays(const m2_plan* pl, int count, int64_t B, int64_t H, int64_t n) {
    return has_time_kernel(pl) && pl->N == 512 && n > 160 && n <= 256 && n % 8 == 0 && B > 16 &&
           count * H * ((B + kRowsPerItem - 1) / kRowsPerItem) >= (n >= 192 ? 445 + (256 - n) * 3 / 2 : 889);
}

int32_t conv_umma(const m2_plan* pl, const Rows* sets, int count, int64_t B, int64_t H, int64_t n, int kf_group, cudaStream_t stream) {
    const int64_t per_set = H * ((B + kRowsPerItem - 1) / kRowsPerItem), items = per_set * count;
    if (items == 0) return M2_OK;
    if (items > 0x3fffffffLL || B > 0x7fffffffLL || H > 0x7fffffffLL) return M2_ERR_UNSUPPORTED;
    alignas(64) UmmaArgs A = {};
    for (int i = 0; i < count; ++i) {
        const Rows& r = sets[i];
        if (!map_rows(&A.x[i], r.x, B, H, n) || !map_rows(&A.y[i], r.y, B, H, n)) return M2_ERR_UNSUPPORTED;
        A.kt[i] = r.kt;
    }
    A.H = (int)H;
    A.n = (int)n;
    A.N = (int)pl->N;
    A.kf_group = kf_group;
    A.per_set = (int)per_set;
    A.items = (int)items;
    static std::atomic<bool> done[64];
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return M2_ERR_CUDA;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool known = dev >= 0 && dev < 64;
    if (!known || !done[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(toeplitz_umma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUmmaSmem) != cudaSuccess) return M2_ERR_CUDA;
        if (known) done[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items < sms ? items : sms));
    cfg.blockDim = dim3(kUmmaThreads);
    cfg.dynamicSmemBytes = kUmmaSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, toeplitz_umma_kernel, A, pl->d_status) != cudaSuccess) return M2_ERR_CUDA;
    pl->last_kernel = "conv_toeplitz_umma";
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2t
