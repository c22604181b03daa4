// Batched GEMM on CTA pairs (tcgen05 cta_group::2):  O[bt][j] = A[j] B[bt][j], a tile of 256 output rows x up to 256 columns per pair.
//
// Serves the column-layout Monarch stages whose blocks fill its tiles of 256 rows (cols_umma.cu has the formulation and the rule) and the
// dense projections of the Hyena layer and the M2-BERT mixer (up to three weights in one launch).  Operands are taken as they lie: A is
// K-major (weights) or M-major (activations [k][m]), B is N-major ([k][n]) or K-major ([n][k]); tensor maps do the rest, so the
// projections read x [positions][channels] without a transposition and the output projection writes that layout.
//
// Why pairs: with a 128 x 256 tile per CTA a K step of 64 brings 48 KB into shared memory for 512 cycles of tensor work, 96 bytes per
// cycle and SM, more than L2 delivers.  A pair's 256 x 256 tile shares B: every CTA loads its 128 rows of A and half of the columns of B,
// 32 KB for the same 512 cycles, and the accumulators (256 columns in each CTA) still fit twice.
// Per CTA: warps 0..7 epilogue (lane quarter w % 4, column half w / 4; each warp stages and stores its own boxes, no barrier among
// them), warp 8 TMA producer, warp 9 of the even CTA issues the UMMAs of the pair.  Both CTAs' loads count on the even CTA's barrier;
// commits signal both.  All waits are bounded.
//
// Measured, one B200 (per launch, cold): three projections 768 x 768 of 32 x 512 positions in one launch 52 us (58 GFLOP) where three
// launches took 27 us each, the output projection 25 us where it took 27 and a 10 us transposition; a stage of the 65536 x 768
// operator (256 blocks of 256 x 256, 233 MB) 50 -> 42 us, the one with the factor (335 MB) 72 -> 57 us once its rows came by TMA
// into the staging area instead of 16 bytes per lane from strided rows.  The projections are bound by the operands' way from L2 (32 KB a
// chunk and SM, of which 44 bytes arrive per cycle: tensor pipe 54 % busy for three projections of 32 x 256 positions, 35 % for one), the
// operator by DRAM (5.5 TB/s).
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>

#include "cols_umma.h"
#include "gemm_pair.h"
#include "ptx_sm100.cuh"
#include "tma_host.h"

namespace m2c {

using namespace sm100;

constexpr int kEpilogueWarps = 8, kPairThreads = 32 * (kEpilogueWarps + 2);
constexpr int kPairStages = 5;
constexpr int P_STAGE = 32768;                        // A [128][64] 16384 | B [64][128] 16384
constexpr int P_OUT = kPairStages * P_STAGE;          // staging: 8 KB per epilogue warp, two boxes [32 rows][64 columns]
constexpr int P_BAR = P_OUT + kEpilogueWarps * 8192;  // full[5], empty[5], acc_full[2], acc_empty[2], tmem ptr, abort flag, factor[8]
constexpr int P_SMEM = P_BAR + 192;
static_assert(P_SMEM <= 232448, "shared memory budget");

struct PairMaps {
    CUtensorMap a[3], b, o[3], k;
};

__device__ __forceinline__ uint32_t map_to_even(uint32_t addr) {   // the same shared-memory offset in the pair's even CTA
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
// copy into this CTA's shared memory that counts on a barrier of the pair's even CTA
__device__ __forceinline__ void pair_load_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
                 "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
                 : "memory");
}
// bar: a shared::cluster address.  The arrival releases this warp's tensor-memory loads (complete: wait::ld, fence::before_thread_sync);
// no generic memory is handed over, which is why the scope of the CTA suffices for the arrival in the other CTA.  65536 x 768 operator, one product: 86 us
// relaxed as with this release, 110 with one at cluster scope, which waits for every store in flight.
__device__ __forceinline__ void pair_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void pair_umma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void pair_commit(uint32_t bar) {   // the barrier at this offset in both CTAs
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
                 "h"((uint16_t)3)
                 : "memory");
}
__device__ __forceinline__ void pair_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

struct PairShape {
    int chunks;            // K / 64
    int rows, cols;        // of one output matrix; rows: per weight
    int otiles, ctiles;    // tiles of 256 rows (all weights together) x nc columns
    int otiles_w;          // ... of one weight
    int nb, tiles;         // blocks per matrix; tiles in all
    int nc;                // columns per tile: 256 or 128
    int a_mmajor, b_kmajor, a_batched;
    int kmul, relu;        // factor K (.) on the result (its rows are those of one output matrix), then ReLU
};

// tile index = ((bt * nb + j) * otiles + ot) * ctiles + ct: pairs running at the same time share a block's operands in L2
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
gemm_pair_kernel(const __grid_constant__ PairMaps maps, const __grid_constant__ PairShape S, int32_t* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x & 1, pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const uint32_t s_base = smem_u32(smem);
    const uint32_t bar_full = s_base + P_BAR, bar_empty = bar_full + 8 * kPairStages, bar_accf = bar_empty + 8 * kPairStages,
                   bar_acce = bar_accf + 16, s_tptr = bar_acce + 16, bar_k = s_tptr + 16;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + P_BAR + 16 * kPairStages + 40);
    if (tid == 0) {
        for (int s = 0; s < kPairStages; ++s) {
            mbar_init(bar_full + 8 * s, 1);
            mbar_init(bar_empty + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_accf + 8 * a, 1);
            mbar_init(bar_acce + 8 * a, 2 * kEpilogueWarps);   // one arrival per epilogue warp of the pair
        }
        for (int w = 0; w < kEpilogueWarps; ++w) mbar_init(bar_k + 8 * w, 1);
        *abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_tptr), "r"((uint32_t)(2 * S.nc)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    pair_sync();   // both CTAs' barriers exist
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the operands may have been written by the kernel before this one
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + P_BAR + 16 * kPairStages + 32);
    const int half = S.nc / 2;
    bool ok = true;

    if (warp == 8) {
        // ---- TMA producer ----------------------------------------------------------------------------------------------
        if (lane == 0) {
            const uint32_t tx = 2u * (16384u + (uint32_t)half * 128u);   // both CTAs' copies of a stage
            const uint32_t full0 = map_to_even(bar_full);
            uint32_t n = 0;
            for (int t = pair; t < S.tiles && ok; t += pairs) {
                const int ct = t % S.ctiles, ot = (t / S.ctiles) % S.otiles, j = (t / (S.ctiles * S.otiles)) % S.nb,
                          bt = t / (S.ctiles * S.otiles * S.nb);
                const CUtensorMap* ma = &maps.a[ot / S.otiles_w];
                const int m0 = (ot % S.otiles_w) * 256 + rank * 128, c0 = ct * S.nc + rank * half, abt = S.a_batched ? bt : 0;
                for (int kc = 0; kc < S.chunks; ++kc, ++n) {
                    const int s = n % kPairStages;
                    if (n >= kPairStages) ok = mbar_wait(bar_empty + 8 * s, ((n / kPairStages) - 1) & 1);   // the UMMAs have read the buffer
                    if (!ok || *abort_flag) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = s_base + s * P_STAGE, sb = sa + 16384, bf = full0 + 8 * s;
                    if (rank == 0) mbar_expect_tx(bar_full + 8 * s, tx);
                    if (S.a_mmajor) {
                        pair_load_4d(sa, ma, m0, kc * 64, j, abt, bf);
                        pair_load_4d(sa + 8192, ma, m0 + 64, kc * 64, j, abt, bf);
                    } else {
                        pair_load_4d(sa, ma, kc * 64, m0, j, abt, bf);
                    }
                    const int bbt = S.a_batched ? 0 : bt;   // one of the two operands is the weight
                    if (S.b_kmajor) {
                        pair_load_4d(sb, &maps.b, kc * 64, c0, j, bbt, bf);
                    } else {
                        for (int q = 0; q < half; q += 64) pair_load_4d(sb + q * 128, &maps.b, c0 + q, kc * 64, j, bbt, bf);
                    }
                }
            }
            // the last stages' commits arrive in this CTA, too: stay until they have
            for (uint32_t i = n > kPairStages ? n - kPairStages : 0; i < n && ok; ++i)
                ok = mbar_wait(bar_empty + 8 * (i % kPairStages), (i / kPairStages) & 1);
        }
    } else if (warp == 9) {
        // ---- UMMA issuer (of the pair) -----------------------------------------------------------------------------------
        if (lane == 0 && rank == 0) {
            const uint32_t idesc = instr_desc_bf16(256, S.nc, S.a_mmajor != 0, S.b_kmajor == 0);
            const uint32_t astep = (S.a_mmajor ? 2048 : 32) >> 4, bstep = (S.b_kmajor ? 32 : 2048) >> 4;   // 16 inputs further on
            // base descriptors; the address field counts 16 bytes (LBO is not used by K-major swizzled operands)
            const uint64_t da0 = smem_desc_sw128(s_base, 8192, 1024), db0 = smem_desc_sw128(s_base + 16384, 8192, 1024);
            uint32_t s = 0, ph = 0;   // stage and phase of the next chunk
            bool ready = false;       // its operands are known to have landed
            int it = 0;
            for (int t = pair; t < S.tiles && ok; t += pairs, ++it) {
                const int acc = it & 1;
                const uint32_t d = tmem + acc * S.nc;
                if (it >= 2) ok = mbar_wait(bar_acce + 8 * acc, ((it >> 1) - 1) & 1);   // both epilogues have read this accumulator
                for (int kc = 0; kc < S.chunks && ok; ++kc) {
                    if (!ready) ok = mbar_wait(bar_full + 8 * s, ph);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t da = da0 + s * (P_STAGE >> 4), db = db0 + s * (P_STAGE >> 4);
                    const uint32_t bar_e = bar_empty + 8 * s;
                    pair_umma(d, da, db, idesc, kc != 0);
                    pair_umma(d, da + astep, db + bstep, idesc, 1);
                    pair_umma(d, da + 2 * astep, db + 2 * bstep, idesc, 1);
                    if (++s == kPairStages) {
                        s = 0;
                        ph ^= 1;
                    }
                    // an issue blocks until the tensor core takes the instruction: the next chunk's barrier is looked at while it works
                    ready = mbar_test(bar_full + 8 * s, ph);
                    pair_umma(d, da + 3 * astep, db + 3 * bstep, idesc, 1);
                    pair_commit(bar_e);
                }
                if (ok) pair_commit(bar_accf + 8 * acc);
            }
        }
    } else {
        // ---- epilogue: accumulator row = lane = output row of this CTA's half; the warp's columns [hc half, hc half + half) of the tile,
        //      64 at a time ----
        const int q = warp & 3, hc = warp >> 2, nbox = half / 64;
        const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16) + hc * half;
        const uint32_t acce0 = map_to_even(bar_acce);
        unsigned char* stg = smem + P_OUT + warp * 8192;
        int it = 0;
        for (int t = pair; t < S.tiles && ok; t += pairs, ++it) {
            const int ct = t % S.ctiles, ot = (t / S.ctiles) % S.otiles, j = (t / (S.ctiles * S.otiles)) % S.nb,
                      bt = t / (S.ctiles * S.otiles * S.nb);
            const int acc = it & 1, o0 = (ot % S.otiles_w) * 256 + rank * 128 + q * 32, c0 = ct * S.nc + hc * half;
            if (lane == 0) {
                tma_store_wait_read0();   // this warp's previous stores have read the staging area
                if (S.kmul) {             // the factor's boxes wait there while the tile's UMMAs run
                    mbar_expect_tx(bar_k + 8 * warp, (uint32_t)nbox * 4096u);
                    for (int bx = 0; bx < nbox; ++bx)
                        tma_load_4d(s_base + P_OUT + warp * 8192 + bx * 4096, &maps.k, c0 + 64 * bx, o0, j, 0, bar_k + 8 * warp);
                }
            }
            ok = mbar_wait(bar_accf + 8 * acc, (it >> 1) & 1);
            if (ok && S.kmul) ok = mbar_wait(bar_k + 8 * warp, it & 1);
            ok = __all_sync(0xffffffffu, ok && *abort_flag == 0);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int bx = 0; bx < 2; ++bx) {
                if (bx >= nbox) break;
#pragma unroll
                for (int hq = 0; hq < 2; ++hq) {
                    float v[32];
#pragma unroll
                    for (int c8 = 0; c8 < 4; ++c8) tmem_ld8(t_lane + acc * S.nc + bx * 64 + (hq * 4 + c8) * 8, v + 8 * c8);
                    tmem_ld_wait();
#pragma unroll
                    for (int c8 = 0; c8 < 4; ++c8) tmem_ld_fence8(v + 8 * c8);
#pragma unroll
                    for (int c8 = 0; c8 < 4; ++c8) {
                        float* w = v + 8 * c8;
                        uint4* cell = reinterpret_cast<uint4*>(stg + bx * 4096 + lane * 128 + (((hq * 4 + c8) ^ (lane & 7)) << 4));
                        if (S.kmul) {
                            const uint4 kp = *cell;
                            const uint32_t kw[4] = {kp.x, kp.y, kp.z, kp.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                w[2 * e] *= __uint_as_float(kw[e] << 16);
                                w[2 * e + 1] *= __uint_as_float(kw[e] & 0xffff0000u);
                            }
                            if (S.relu) {
#pragma unroll
                                for (int e = 0; e < 8; ++e) w[e] = fmaxf(w[e], 0.f);
                            }
                        }
                        *cell = make_uint4(pack2(w[0], w[1]), pack2(w[2], w[3]), pack2(w[4], w[5]), pack2(w[6], w[7]));
                    }
                }
            }
            tc_fence_before();
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                pair_arrive(acce0 + 8 * acc);   // this warp has read its part of the accumulator
                if (o0 < S.rows)                // (rows and columns past the matrix are clipped by the tensor map)
                    for (int bx = 0; bx < nbox; ++bx)
                        if (c0 + 64 * bx < S.cols)
                            tma_store_4d(&maps.o[ot / S.otiles_w], s_base + P_OUT + warp * 8192 + bx * 4096, c0 + 64 * bx, o0, j, bt);
                tma_store_commit();
            }
        }
        if (lane == 0) tma_store_wait_read0();   // the staging area dies with the CTA
    }
    if (!ok && lane == 0) {
        *abort_flag = 1;
        atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);   // copies issued before the wait ran out have landed by then
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    pair_sync();   // no signal to a CTA that has left
    if (warp == 9) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * S.nc)) : "memory");
}

static cudaError_t pair_prepare() {
    static std::atomic<bool> done[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(gemm_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, P_SMEM);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(true, std::memory_order_release);
    return e;
}

static bool map4(CUtensorMap* m, const PairTensor& t, uint32_t b0, uint32_t b1) {
    const cuuint64_t gdim[4] = {(cuuint64_t)t.n0, (cuuint64_t)t.n1, (cuuint64_t)t.nj, (cuuint64_t)t.nbt};
    const cuuint64_t gstr[3] = {(cuuint64_t)t.s1 * 2, (cuuint64_t)(t.nj > 1 ? t.sj : t.s1) * 2, (cuuint64_t)(t.nbt > 1 ? t.sbt : t.s1) * 2};
    const cuuint32_t box[4] = {b0, b1, 1, 1};
    return tma_host::encode_sw128_bf16(m, t.p, 4, gdim, gstr, box);
}

int32_t gemm_pair(const m2_plan* pl, const PairGemm& g, cudaStream_t stream) {
    if (pair_prepare() != cudaSuccess) return M2_ERR_CUDA;
    const int64_t rows = g.rows, cols = g.cols;
    PairShape S = {};
    S.nc = cols > 128 ? 256 : 128;
    S.chunks = (int)(g.k / 64);
    S.rows = (int)rows;
    S.cols = (int)cols;
    S.otiles_w = (int)((rows + 255) / 256);
    S.otiles = S.otiles_w * g.weights;
    S.ctiles = (int)((cols + S.nc - 1) / S.nc);
    S.nb = (int)g.o[0].nj;
    S.a_mmajor = g.a_mmajor;
    S.b_kmajor = g.b_kmajor;
    S.a_batched = g.a_batched;
    S.kmul = g.kmul.p != nullptr;
    S.relu = g.relu;
    const int64_t tiles = g.o[0].nbt * S.nb * S.otiles * S.ctiles;
    if (tiles > 0x7fffffffLL) return M2_ERR_UNSUPPORTED;
    if (tiles == 0) return M2_OK;
    S.tiles = (int)tiles;
    alignas(64) PairMaps maps;
    for (int w = 0; w < 3; ++w) {
        const int v = w < g.weights ? w : 0;
        if (!map4(&maps.a[w], g.a[v], 64, g.a_mmajor ? 64 : 128) || !map4(&maps.o[w], g.o[v], 64, 32)) return M2_ERR_UNSUPPORTED;
    }
    if (!map4(&maps.k, g.kmul.p ? g.kmul : g.o[0], 64, 32)) return M2_ERR_UNSUPPORTED;
    if (!map4(&maps.b, g.b, 64, g.b_kmajor ? (uint32_t)(S.nc / 2) : 64)) return M2_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t most = sms / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * (tiles < most ? tiles : most)));
    cfg.blockDim = dim3(kPairThreads);
    cfg.dynamicSmemBytes = P_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, gemm_pair_kernel, maps, S, pl->d_status) != cudaSuccess) return M2_ERR_CUDA;
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2c
