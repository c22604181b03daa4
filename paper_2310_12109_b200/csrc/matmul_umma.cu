// Tensor-core order-2 Monarch matmul for 64 x 64 blocks (N = 4096), bf16 in / fp32 accumulate / bf16 out.
//
//   y[t][k2*64 + k1] = sum_{n2} L[k1][k2][n2] * sum_{n1} R[n2][k1][n1] * x[t][n1*64 + n2]      (Sec. 3.1)
//
// Both block-diagonal factors are batches of 64 independent GEMMs [tokens x 64] x [64 x 64]; the batch
// index is the CONTIGUOUS index of the data each factor reads (n2 for R, k1 for L after the middle
// permutation), so neither operand of a tensor-core GEMM can be taken from memory as it lies.  The two
// factors therefore run as two passes that exchange the intermediate through a caller workspace.  Two
// generations of pass kernels live in this file:
//
//   monarch64_fwd_kernel<1|2>   the forward path (further down): 32 tokens x 16 blocks per item, 32-byte pieces,
//                               weights resident, loading / draining / issuing warps.
//   monarch64_pass_kernel<1|2>  128 tokens x 8 blocks per CTA, 16-byte pieces (described next): serves inputs that are
//                               only 16-byte aligned; its workspace is z[token tile][n2 / 8][k1][t % 128][n2 % 8]:
//
//   pass 1 (R): a CTA owns 128 tokens x 8 consecutive n2.  Threads read 16-byte pieces of x (8 values of
//               n2 for one (t, n1)), transpose 8 x 8 blocks in registers (the permutation P) and write the
//               K-major, 128-byte-swizzled UMMA operand A_{n2}[t][n1]; 8 UMMA groups (M = 128 tokens,
//               N = 64 = k1, K = 64 = n1) fill the 512 TMEM columns; the epilogue gathers, for every k1,
//               the 8 values of n2 from the 8 accumulators as one 16-byte piece (the permutation P^T); the
//               CTA's pieces [k1][t][16 B] are its slab of z and are stored from registers, 512 bytes per warp.
//   pass 2 (L): a CTA owns 128 tokens x 8 consecutive k1; eight bulk copies bring [n2 / 8][k1 % 8][t][16 B] into shared
//               memory, which IS the K-major operand of every k1 without swizzle (core matrix = 8 tokens x 16 bytes,
//               next K chunk 16 KB further); same UMMAs with L's blocks; the epilogue stages 16-byte pieces of
//               y[t][k2][k1] and one dimension-permuting TMA store scatters them (the last P).
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstring>

#include "generic_kernels.h"
#include "matmul_umma.h"
#include "ptx_sm100.cuh"
#include "tma_host.h"

namespace m2mm {

using namespace sm100;

constexpr int kThreads = 512;
constexpr int kTileT = 128;   // tokens per CTA
constexpr int kGroup = 8;     // blocks per CTA
constexpr int OFF_A = 0;                   // 8 operands [128 t][64] bf16, swizzled   131072
constexpr int OFF_B = 131072;              // 8 weight blocks [64][64] bf16, swizzled   65536
constexpr int OFF_BAR = 196608;            // bar_mma, tmem ptr, bar_in
constexpr int SMEM_BYTES = OFF_BAR + 64;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit_wait() {
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(map), "r"(src), "r"(c0),
                 "r"(c1), "r"(c2)
                 : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
                 "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void* gdst, uint32_t ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(ssrc), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// byte offset of 16-byte chunk kc of row r in a K-major operand with 128-byte rows and the 128B swizzle
__device__ __forceinline__ uint32_t sw_off(int r, int kc) { return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((kc ^ (r & 7)) << 4)); }

// PASS 1: in = x[T][64 n1][64 n2], W = R[n2][k1][n1], out = z[T][64 k1][64 n2]
// PASS 2: in = z[T][64 k1][64 n2], W = L[k1][k2][n2], out = y[T][64 k2][64 k1]
template <int PASS>
__global__ void __launch_bounds__(kThreads, 1)
monarch64_pass_kernel(const __nv_bfloat16* __restrict__ in, const __nv_bfloat16* __restrict__ W,
                      const __grid_constant__ CUtensorMap map_out, __nv_bfloat16* __restrict__ zout, long long T,
                      int32_t* __restrict__ status, const __nv_bfloat16* __restrict__ Kmul, long long Hk, int relu) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x;
    const int wg = tid >> 7, t = tid & 127, warp = t >> 5;
    const uint32_t s_base = smem_u32(smem);
    const uint32_t bar_mma = s_base + OFF_BAR, s_tptr = s_base + OFF_BAR + 16, bar_in = s_base + OFF_BAR + 24;
    // the 8 CTAs that share the 128-byte lines of one token tile are neighbours in launch order, so the
    // 16-byte pieces of a line are fetched / written while the line is still in L2
    const long long t0 = (long long)blockIdx.y * kTileT;
    const int grp = blockIdx.x;   // which 8 consecutive blocks (n2 in pass 1, k1 in pass 2)

    if (tid == 0) {
        mbar_init(bar_mma, 1);
        mbar_init(bar_in, 1);
        fence_barrier_init();
    }
    if (tid < 32) tmem_alloc(s_tptr, 512);
    // Programmatic dependent launch: the next kernel's CTAs may take over SMs as this grid's CTAs leave them.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // weight blocks -> swizzled K-major B operands ([64 out][64 in], rows of 128 bytes)
    for (int c = tid; c < kGroup * 64 * 8; c += kThreads) {
        const int kc = c & 7, o = (c >> 3) & 63, bl = c >> 9;
        cp_async16(s_base + OFF_B + bl * 8192 + sw_off(o, kc), W + ((size_t)(grp * kGroup + bl) * 64 + o) * 64 + kc * 8, 16u);
    }
    // The weights are the caller's and were complete before this call; everything else (pass 1's z for pass 2, the
    // producer of x, earlier readers of the buffers written here) is awaited now.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (PASS == 1) {
        // unit = (token tt, group g of 8 consecutive n1): 8 loads of 16 bytes (8 values of n2 each), an 8 x 8
        // transpose in registers, 8 stores (one per n2) of the 8 n1 values = chunk g of row tt of A_{n2}
#pragma unroll 1
        for (int u = tid; u < kTileT * 8; u += kThreads) {
            const int g = u & 7, tt = u >> 3;
            uint4 v[8];
            const bool live = t0 + tt < T;
            const uint4* src = reinterpret_cast<const uint4*>(in + (size_t)(t0 + tt) * 4096 + (size_t)(8 * g) * 64 + grp * 8);
#pragma unroll
            for (int i = 0; i < 8; ++i) {   // cached in L2 only: the other half of every 32-byte sector belongs to another SM
                v[i] = make_uint4(0u, 0u, 0u, 0u);
                if (live)
                    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[i].x), "=r"(v[i].y), "=r"(v[i].z), "=r"(v[i].w) : "l"(src + i * 8));
            }
            const uint32_t* w = reinterpret_cast<const uint32_t*>(v);   // w[i*4 + j]: n1 = 8g+i, n2 = 2j, 2j+1
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint4 lo, hi;
                lo.x = prmt(w[0 * 4 + j], w[1 * 4 + j], 0x5410); hi.x = prmt(w[0 * 4 + j], w[1 * 4 + j], 0x7632);
                lo.y = prmt(w[2 * 4 + j], w[3 * 4 + j], 0x5410); hi.y = prmt(w[2 * 4 + j], w[3 * 4 + j], 0x7632);
                lo.z = prmt(w[4 * 4 + j], w[5 * 4 + j], 0x5410); hi.z = prmt(w[4 * 4 + j], w[5 * 4 + j], 0x7632);
                lo.w = prmt(w[6 * 4 + j], w[7 * 4 + j], 0x5410); hi.w = prmt(w[6 * 4 + j], w[7 * 4 + j], 0x7632);
                *reinterpret_cast<uint4*>(smem + OFF_A + (2 * j) * 16384 + sw_off(tt, g)) = lo;
                *reinterpret_cast<uint4*>(smem + OFF_A + (2 * j + 1) * 16384 + sw_off(tt, g)) = hi;
            }
        }
    } else if (tid == 0) {
        // z block (token tile, n2 group kc, k1 group grp) = [k1 % 8][t][8 n2] = 16 KB: chunk kc of every operand row
        mbar_expect_tx(bar_in, 8 * 16384);
        const unsigned char* zb = reinterpret_cast<const unsigned char*>(in) + (size_t)blockIdx.y * (8 * 131072) + (size_t)grp * 16384;
        for (int kc = 0; kc < 8; ++kc) bulk_load(s_base + OFF_A + kc * 16384, zb + (size_t)kc * 131072, 16384, bar_in);
    }
    cp_async_commit_wait();
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + OFF_BAR + 16);

    if (tid < 32 && elect_one()) {
        constexpr uint32_t IDESC = instr_desc_bf16(128, 64, false, false);
        bool in_ok = true;
        if (PASS == 2) in_ok = mbar_wait(bar_in, 0);
        if (in_ok) {
#pragma unroll 1
            for (int bl = 0; bl < kGroup; ++bl)
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    umma_f16(tmem + bl * 64,
                             PASS == 1 ? smem_desc_sw128(s_base + OFF_A + bl * 16384 + s * 32, 16, 1024)
                                       : smem_desc(s_base + OFF_A + bl * 2048 + s * 32768, 16384, 128),
                             smem_desc_sw128(s_base + OFF_B + bl * 8192 + s * 32, 16, 1024), IDESC, s > 0);
        }
        umma_commit(bar_mma);   // (with no UMMA issued it completes at once; the missing input is reported below)
        if (!in_ok) atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
    }
    const bool ok = mbar_wait(bar_mma, 0);
    tc_fence_after();
    // epilogue: lane = token; warpgroup wg takes output columns [16 wg, 16 wg + 16); for every output index o the 8
    // accumulators give the 8 consecutive block indices -> one 16-byte piece.  The pieces are staged in the (now free)
    // operand buffer with consecutive lanes writing to different banks, then leave through the copy engine:
    //   pass 1: the pieces [k1][t][16 B] are this CTA's contiguous slab of z and go straight from registers to global
    //           memory (a warp's 32 tokens are 512 contiguous bytes);
    //   pass 2: y[t][k2][k1]     -- staged as [k2][t][16 B]; one TMA store whose tensor map lists the dimensions as
    //                               (k1, t, k2) scatters the pieces (rows past T are clipped by the map).
    unsigned char* zslab = PASS == 1 ? reinterpret_cast<unsigned char*>(zout) + ((size_t)blockIdx.y * 8 + grp) * 131072 : nullptr;
    if (ok) {
        const uint32_t t_lane = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int gk = 0; gk < 2; ++gk) {
            const int o0 = 16 * wg + 8 * gk;
            float v[8][8];
#pragma unroll
            for (int bl = 0; bl < 8; ++bl) tmem_ld8(t_lane + bl * 64 + o0, v[bl]);
            tmem_ld_wait();
#pragma unroll
            for (int bl = 0; bl < 8; ++bl) tmem_ld_fence8(v[bl]);
            if (PASS == 2 && Kmul != nullptr && t0 + t < T) {
                // y = sigma(K (.) M x) (first half of the M2 operator, Eq. 2): the 8 accumulators of one kk are the 8
                // consecutive k1 of output index k2*64 + k1 -> one 16-byte piece of the kernel row
                const __nv_bfloat16* krow = Kmul + (size_t)((t0 + t) % Hk) * 4096 + 8 * grp;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint4 kp = *reinterpret_cast<const uint4*>(krow + (o0 + kk) * 64);
                    const uint32_t kw[4] = {kp.x, kp.y, kp.z, kp.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        float a = v[2 * q][kk] * __uint_as_float(kw[q] << 16);
                        float b = v[2 * q + 1][kk] * __uint_as_float(kw[q] & 0xffff0000u);
                        v[2 * q][kk] = relu ? fmaxf(a, 0.f) : a;
                        v[2 * q + 1][kk] = relu ? fmaxf(b, 0.f) : b;
                    }
                }
            }
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const uint4 p = make_uint4(pack_bf16(v[0][kk], v[1][kk]), pack_bf16(v[2][kk], v[3][kk]),
                                           pack_bf16(v[4][kk], v[5][kk]), pack_bf16(v[6][kk], v[7][kk]));
                if (PASS == 1)   // z slab [k1][token][16 B]: a warp's 32 tokens are 512 contiguous bytes, stored as they are
                    *reinterpret_cast<uint4*>(zslab + (o0 + kk) * 2048 + t * 16) = p;
                else             // [k2][token][16 B], scattered to y by the TMA store below
                    *reinterpret_cast<uint4*>(smem + OFF_A + (o0 + kk) * 2048 + t * 16) = p;
            }
        }
    }
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (PASS == 2 && tid == 0 && ok) {
        tma_store_3d(&map_out, s_base + OFF_A, 8 * grp, (int)t0, 0);
        tma_store_commit();
        tma_store_wait_read0();   // the staging buffer dies with the CTA
    }
    __syncthreads();
    if (!ok && tid == 0) atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
    if (tid < 32) tmem_dealloc(tmem, 512);
}

bool covered(const m2_plan* pl);
int64_t workspace_bytes(const m2_plan* pl, int64_t T);

// ---- the forward passes: 32 tokens x 16 blocks per item ------------------------------------------------------------------
//
// The cost of both passes is the number of memory requests for the pieces of x (pass 1) and of y (pass 2) that a CTA owning
// g consecutive blocks touches: 2 g bytes of every 128-byte line.  With g = 16 a piece is a whole 32-byte sector.  An SM takes
// such requests at a fixed rate (and a warp that issues them is blocked while they queue), so everything else a tile needs
// runs underneath them, in other warps:
//
//   UMMA         the WEIGHT block is the A operand (M = 64 output indices, K = 64) and the tile's data the B operand (N = 32
//                tokens): D_b[out][t].  Row r of an M = 64 accumulator lives in TMEM lane (r % 16) + 32 (r / 16), so blocks
//                8..15 sit at lane offset 16 in the columns of blocks 0..7: a tile's 16 accumulators take 256 columns, and
//                the 512 columns hold TWO tiles -- the UMMAs of tile i run while the accumulators of tile i - 1 are drained.
//   weights      all 16 blocks of the CTA's group stay in shared memory (128 KB, one TMA tile per block, 128-byte swizzle =
//                the K-major operand image); the 16 operands of a 32-token tile take the other 64 KB.
//   roles        warps 0..7 load (global -> registers -> operand buffer), warps 8..15 drain (TMEM -> registers -> global),
//                lane 0 of warps 16 and 17 issues 8 blocks each (32 UMMAs, ~60 cycles of the thread's time per instruction,
//                about what the tensor core needs for them).  They meet only through mbarriers.
//   workspace    z[32-token tile][n2 / 16][t % 32][k1][n2 % 16]: 32-byte pieces with k1 running fastest.  In pass 1 lane l of a
//                draining warp holds output index k1 = 16 q + l % 16 of blocks 8 (l / 16) .. + 7, i.e. 16 bytes of a piece, and a
//                warp store is 512 contiguous bytes; in pass 2 the CTA (tile, k1 group) reads, for every (n2 / 16, t), 16 pieces
//                = 512 contiguous bytes, and a piece is 32 bytes of row t of the K-major operand of its block as it lies.
//   pass 1 in    one (token, 8 consecutive n1) per loading thread: 8 loads of 32 bytes, a 16 x 8 transpose in registers (PRMT;
//                this is P), 16 stores of 16 bytes into the swizzled operands B_{n2}[t][n1].
//   pass 2 out   y[t][k2][16 k1]: a thread's 8 accumulators of one token are 16 bytes, the lane 16 further holds the other half
//                of the sector.  Each draining warp stages [4 tokens][its 16 k2][32 B] in shared memory (the 32-byte-swizzled
//                image of a TMA box: no bank conflicts) and lane 0 sends it off with one tensor store (the last P): the 2048
//                sectors a tile scatters over 2048 lines never pass through the load/store unit, whose request rate is
//                what the loads need; rows past T are clipped by the tensor map.
constexpr int kTok = 32;                      // tokens per item
constexpr int kGroup2 = 16;                   // blocks per CTA
constexpr int F_OFF_A = 0;                    // 16 operands [32 t][64] bf16, swizzled rows of 128 bytes      65536
constexpr int F_OFF_W = 65536;                // 16 weight blocks [64][64] bf16, swizzled                     131072
constexpr int kLoadWarps = 8, kDrainWarps = 8, kIssueWarps = 2;
constexpr int F_OFF_ST = F_OFF_W + kGroup2 * 8192;    // pass 2: per draining warp two staging buffers [4 t][16 k2][32 B]  32768
constexpr int F_OFF_BAR = F_OFF_ST + kDrainWarps * 4096;   // bar_w, bar_mma[2], tmem ptr, abort flag, bar_opnd, bar_tfree[2]
constexpr int F_SMEM_BYTES = F_OFF_BAR + 64;
constexpr int kFwdThreads = 32 * (kLoadWarps + kDrainWarps + kIssueWarps);
constexpr size_t kTileBytes = (size_t)kTok * 8192;    // a tile of x, z or y
static_assert(F_SMEM_BYTES <= 232448, "shared-memory budget of the forward passes");

// 8 pieces of 16 consecutive block indices, one per 128-byte line; cached in L2 only: the rest of every line belongs to other SMs.
// HALVES: rows that are only 16-byte aligned come as two halves.
template <bool HALVES>
__device__ __forceinline__ void load_pieces(uint32_t (&w)[8][8], const unsigned char* src, bool live) {
    const bool whole = !HALVES || (reinterpret_cast<uintptr_t>(src) & 31u) == 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (live && whole) {
            asm volatile("ld.global.cg.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(w[i][0]), "=r"(w[i][1]), "=r"(w[i][2]), "=r"(w[i][3]), "=r"(w[i][4]), "=r"(w[i][5]), "=r"(w[i][6]), "=r"(w[i][7])
                         : "l"(src + i * 128));
        } else if (live) {
#pragma unroll
            for (int m = 0; m < 8; m += 4)
                asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(w[i][m]), "=r"(w[i][m + 1]), "=r"(w[i][m + 2]), "=r"(w[i][m + 3])
                             : "l"(src + i * 128 + m * 4));
        } else {
#pragma unroll
            for (int m = 0; m < 8; ++m) w[i][m] = 0u;
        }
    }
}
// the 16 x 8 transpose in registers (this is P): 16 bytes = 8 consecutive values of the contracted index of one (token, block), into
// the swizzled operands [token][64] of 16 blocks, 4 KB apart
__device__ __forceinline__ void store_pieces(const uint32_t (&w)[8][8], unsigned char* dst) {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
        uint4 lo, hi;
        lo.x = prmt(w[0][m], w[1][m], 0x5410); hi.x = prmt(w[0][m], w[1][m], 0x7632);
        lo.y = prmt(w[2][m], w[3][m], 0x5410); hi.y = prmt(w[2][m], w[3][m], 0x7632);
        lo.z = prmt(w[4][m], w[5][m], 0x5410); hi.z = prmt(w[4][m], w[5][m], 0x7632);
        lo.w = prmt(w[6][m], w[7][m], 0x5410); hi.w = prmt(w[6][m], w[7][m], 0x7632);
        *reinterpret_cast<uint4*>(dst + (2 * m) * 4096) = lo;
        *reinterpret_cast<uint4*>(dst + (2 * m + 1) * 4096) = hi;
    }
}

// PASS 1: in = x[T][64 n1][64 n2], weights R[n2][k1][n1], out = workspace z
// PASS 2: in = workspace z, weights L[k1][k2][n2], out = y[T][64 k2][64 k1] (optionally sigma(K (.) y))
//
// BWD (the products of the backward pass; a variant of its own because the run-time choices cost the forward pass 2 %): with wt every
// weight block is used transposed -- the block as it lies in shared memory is then an M-major operand instead of a K-major one, nothing is
// moved --, and `in` of pass 1 may be on a 16-byte boundary only.
//
// Persistent: CTA c of a grid that is a multiple of 4 walks the items c, c + grid, .. of (token tile, block group) pairs numbered
// group-fastest, so its block group is c % 4 for good (the weights stay) and the 4 CTAs that share a tile's lines work on it at
// the same time.  Tile i of a CTA uses accumulator set i % 2:
//   loading warps   wait for the UMMAs of tile i - 1 (operand buffer free), write tile i's operands from their registers, arrive on
//                   bar_opnd, request tile i + 1;
//   issuing threads wait for bar_opnd (operands of tile i) and bar_tfree[i % 2] (set drained of tile i - 2), issue, commit to
//                   bar_mma[i % 2];
//   draining warps  wait for bar_mma[i % 2], move the set to global memory, arrive on bar_tfree[i % 2].
template <int PASS, bool BWD>
__global__ void __launch_bounds__(kFwdThreads, 1)
monarch64_fwd_kernel(const __nv_bfloat16* __restrict__ in, const __grid_constant__ CUtensorMap map_w,
                     const __grid_constant__ CUtensorMap map_y, __nv_bfloat16* __restrict__ out, long long T,
                     int32_t* __restrict__ status, const __nv_bfloat16* __restrict__ Kmul, long long Hk, int relu, int selftest, int wt) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t s_base = smem_u32(smem);
    const uint32_t bar_w = s_base + F_OFF_BAR, bar_mma = bar_w + 8, s_tptr = bar_w + 24, bar_opnd = bar_w + 40, bar_tfree = bar_w + 48;
    // selftest: the issuing threads issue and commit nothing and every wait for them gives up after a few polls, so that all
    // roles leave through their abort paths with nothing of theirs in flight
    const uint32_t wlim = selftest ? 64u : (1u << 22);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + F_OFF_BAR + 32);
    const int grp = blockIdx.x & 3;                                   // which 16 consecutive blocks (n2 in pass 1, k1 in pass 2)
    const long long ntiles = (T + kTok - 1) / kTok, nitems = 4 * ntiles;
    long long item = blockIdx.x;
    // pass 2 walks the tiles from the last to the first: what pass 1 wrote last is what the L2 still holds
    auto tile_of = [&](long long it) { return PASS == 1 ? it >> 2 : ntiles - 1 - (it >> 2); };
    if (tid == 0) {
        mbar_init(bar_w, 1);
        mbar_init(bar_mma, kIssueWarps);       // one arrival per issuing thread
        mbar_init(bar_mma + 8, kIssueWarps);
        mbar_init(bar_opnd, kLoadWarps);       // one arrival per loading warp
        mbar_init(bar_tfree, kDrainWarps);     // one arrival per draining warp
        mbar_init(bar_tfree + 8, kDrainWarps);
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&map_w);
        if (PASS == 2) prefetch_tensormap(&map_y);
    }
    if (warp == 2) tmem_alloc(s_tptr, 512);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();   // barriers initialised before anyone arms them
    // the weights are the caller's and were complete before this call
    if (tid == 32) {
        mbar_expect_tx(bar_w, kGroup2 * 8192);
        for (int b = 0; b < kGroup2; ++b) tma_load_2d(s_base + F_OFF_W + b * 8192, &map_w, 0, (grp * kGroup2 + b) * 64, bar_w);
    }
    // this CTA's quarter of a tile's lines, pulled towards L2 as whole lines well before the pieces are read (the four CTAs that
    // share a tile ask for a quarter each).  L2 is where the previous kernel's writes land, so nothing stale can be fetched.
    auto prefetch_item = [&](long long it) {
        if (it < nitems) {
            const long long t0p = tile_of(it) * kTok;
            const long long rows = PASS == 2 || T - t0p >= kTok ? kTok : T - t0p;   // (whole tiles of the workspace exist)
            const long long share = rows * 8192 / 4;
            bulk_prefetch_l2(reinterpret_cast<const unsigned char*>(in) + t0p * 8192 + grp * share, (uint32_t)share);
        }
    };
    if (tid == 33) {
        prefetch_item(item);
        prefetch_item(item + gridDim.x);
    }
    // everything else (pass 1's z for pass 2, the producer of x, earlier readers of the buffers written here) is awaited now
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + F_OFF_BAR + 24);
    uint32_t it_n = 0;        // tiles begun: tile it_n of this CTA uses accumulator set it_n % 2 and phase it_n / 2 of that set's barriers
    bool ok = true;
    auto timed_out = [&]() {
        atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
        *abort_flag = 1;
    };

    if (warp < kLoadWarps) {
        // ---- loading warps: the 2048 pieces of an item, 8 per thread ----
        // Pass 1: (token tid / 8, n1 = 8 (tid % 8) + i), a piece = 16 consecutive n2; the quarter-warp that shared memory serves a
        // 16-byte store in writes the 8 chunks of one row: no bank conflicts.
        // Pass 2: (token 16 (warp / 4) + 8 (i / 4) + lane % 8, k1 = 4 (warp % 4) + lane / 8 of the group, n2 / 16 = i % 4): a warp reads 8
        // whole lines, and a quarter-warp stores to 8 different rows.
        const int t_in = PASS == 1 ? tid >> 3 : 16 * (warp >> 2) + (lane & 7);
        const int sub = PASS == 1 ? tid & 7 : 4 * (warp & 3) + (lane >> 3);
        uint32_t w[8][8];
        auto load_in = [&](long long it) {
            const long long tile = tile_of(it);
            if (PASS == 1) {
                const bool live = tile * kTok + t_in < T;
                const unsigned char* src =
                    reinterpret_cast<const unsigned char*>(in) + (size_t)(tile * kTok + t_in) * 8192 + (size_t)(8 * sub) * 128 + grp * 32;
                load_pieces<BWD>(w, src, live);
            } else {   // whole tiles of the workspace were written
                const unsigned char* src =
                    reinterpret_cast<const unsigned char*>(in) + (size_t)tile * kTileBytes + (size_t)t_in * 2048 + (size_t)(16 * grp + sub) * 32;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    asm volatile("ld.global.cg.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                                 : "=r"(w[i][0]), "=r"(w[i][1]), "=r"(w[i][2]), "=r"(w[i][3]), "=r"(w[i][4]), "=r"(w[i][5]), "=r"(w[i][6]), "=r"(w[i][7])
                                 : "l"(src + (size_t)(i & 3) * 65536 + (size_t)(i >> 2) * (8 * 2048)));
            }
        };
        auto store_opnd = [&]() {
            if (PASS == 1) {
                store_pieces(w, smem + F_OFF_A + sw_off(t_in, sub));
            } else {           // a piece is 32 bytes of row t of block k1's operand as it lies
                unsigned char* dst = smem + F_OFF_A + sub * 4096;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int t = t_in + 8 * (i >> 2), c = 2 * (i & 3);
                    *reinterpret_cast<uint4*>(dst + sw_off(t, c)) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
                    *reinterpret_cast<uint4*>(dst + sw_off(t, c + 1)) = make_uint4(w[i][4], w[i][5], w[i][6], w[i][7]);
                }
            }
        };
        if (item < nitems) load_in(item);
#pragma unroll 1
        for (; item < nitems; item += gridDim.x, ++it_n) {
            if (__any_sync(~0u, *abort_flag != 0)) break;
            // the UMMAs of the previous tile have read the operand buffer
            if (it_n > 0) ok = __all_sync(~0u, mbar_wait(bar_mma + 8 * ((it_n - 1u) & 1u), ((it_n - 1u) >> 1) & 1u, wlim));
            if (!ok) break;
            store_opnd();
            fence_proxy_async();   // operands visible to the tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_opnd);
            // the next tile's pieces are requested now and arrive while this one is computed
            if (item + gridDim.x < nitems) load_in(item + gridDim.x);
            if (tid == 33) prefetch_item(item + 2 * (long long)gridDim.x);
        }
        if (!ok && lane == 0) timed_out();
    } else if (warp < kLoadWarps + kDrainWarps) {
        // ---- draining warps: lane l of lane quarter q = warp % 4 holds output index 16 q + (l & 15) of blocks 8 (l >> 4) .. + 7; the two
        // warps of a quarter split the 32 tokens.  For every token the 8 accumulators of a thread are 8 consecutive block indices:
        // one 16-byte piece. ----
        const int q = warp & 3, c2 = (warp - kLoadWarps) >> 2, r = 16 * q + (lane & 15), set = lane >> 4;
#pragma unroll 1
        for (; item < nitems; item += gridDim.x, ++it_n) {
            if (__any_sync(~0u, *abort_flag != 0)) break;
            const uint32_t p = it_n & 1u;
            const long long tile = tile_of(item), t0 = tile * kTok + 16 * c2;
            ok = __all_sync(~0u, mbar_wait(bar_mma + 8 * p, (it_n >> 1) & 1u, wlim));
            if (!ok) break;
            tc_fence_after();
            const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16) + p * 256u + 16u * c2;
            // pass 1: z[tile][grp][t][k1][32 B], straight from registers, 512 contiguous bytes per warp store
            unsigned char* dst = reinterpret_cast<unsigned char*>(out) + (size_t)tile * kTileBytes + (size_t)grp * 65536 + (size_t)(16 * c2) * 2048 + r * 32 + set * 16;
            // pass 2: this warp's staging buffers; chunk (16 bytes) index XOR bit 7 of the address = the 32-byte swizzle of the box
            const uint32_t st_warp = F_OFF_ST + (uint32_t)(warp - kLoadWarps) * 4096u;
            const uint32_t st_lane = (uint32_t)(lane & 15) * 32u + (uint32_t)((set ^ ((lane >> 2) & 1)) << 4);
#pragma unroll 1
            for (int h = 0; h < 4; ++h) {
                float v[8][4];
#pragma unroll
                for (int bl = 0; bl < 8; ++bl) tmem_ld4(t_lane + bl * 32 + 4 * h, v[bl]);
                if (PASS == 2) {   // the buffer of two rounds ago has been read by its store
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    __syncwarp();
                }
                tmem_ld_wait();
#pragma unroll
                for (int bl = 0; bl < 8; ++bl) tmem_ld_fence4(v[bl]);
                if (PASS == 2 && Kmul != nullptr) {
                    // y = sigma(K (.) M x) (first half of the M2 operator, Eq. 2): the 8 accumulators of one token are 8 consecutive k1
                    // -> one 16-byte piece of the kernel row
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const long long t = t0 + 4 * h + kk;
                        if (t < T) {
                            const uint4 kp = *reinterpret_cast<const uint4*>(Kmul + (size_t)(t % Hk) * 4096 + r * 64 + 16 * grp + 8 * set);
                            const uint32_t kw[4] = {kp.x, kp.y, kp.z, kp.w};
#pragma unroll
                            for (int pp = 0; pp < 4; ++pp) {
                                float a = v[2 * pp][kk] * __uint_as_float(kw[pp] << 16);
                                float bb = v[2 * pp + 1][kk] * __uint_as_float(kw[pp] & 0xffff0000u);
                                v[2 * pp][kk] = relu ? fmaxf(a, 0.f) : a;
                                v[2 * pp + 1][kk] = relu ? fmaxf(bb, 0.f) : bb;
                            }
                        }
                    }
                }
                unsigned char* stg = smem + st_warp + (uint32_t)(h & 1) * 2048u + st_lane;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint4 pk = make_uint4(pack_bf16(v[0][kk], v[1][kk]), pack_bf16(v[2][kk], v[3][kk]),
                                                pack_bf16(v[4][kk], v[5][kk]), pack_bf16(v[6][kk], v[7][kk]));
                    if (PASS == 1)   // whole tiles of the workspace are written (rows past T are zeros)
                        *reinterpret_cast<uint4*>(dst + (size_t)(4 * h + kk) * 2048) = pk;
                    else
                        *reinterpret_cast<uint4*>(stg + kk * 512) = pk;
                }
                if (PASS == 2) {
                    fence_proxy_async();   // staged rows visible to the copy engine
                    __syncwarp();
                    if (lane == 0 && t0 + 4 * h < T) {   // (a box that starts past T has nothing to store)
                        tma_store_3d(&map_y, s_base + st_warp + (uint32_t)(h & 1) * 2048u, 16 * grp, 16 * q, (int)(t0 + 4 * h));
                        tma_store_commit();
                    }
                }
            }
            // the set may be overwritten: this warp's TMEM loads are complete
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tfree + 8 * p);
        }
        if (PASS == 2 && lane == 0) tma_store_wait_all0();   // this thread's stores are complete before shared memory goes away
        if (!ok && lane == 0) timed_out();
    } else if (elect_one()) {
        // ---- issuing threads ----
        const uint32_t idesc = instr_desc_bf16(64, kTok, BWD && wt != 0, false);
        const uint64_t wstep = BWD && wt ? 2048 >> 4 : 32 >> 4;   // 16 inputs: rows of the block as it lies, or 32 bytes of a row
        constexpr int kPer = kGroup2 / kIssueWarps;
        const int b0 = (warp - kLoadWarps - kDrainWarps) * kPer;
        ok = mbar_wait(bar_w, 0);
#pragma unroll 1
        for (; item < nitems && ok && *abort_flag == 0; item += gridDim.x, ++it_n) {
            const uint32_t p = it_n & 1u;
            ok = mbar_wait(bar_opnd, p, wlim);
            if (ok && it_n >= 2) ok = mbar_wait(bar_tfree + 8 * p, ((it_n - 2u) >> 1) & 1u, wlim);
            if (!ok) break;
            if (selftest) continue;
            tc_fence_after();
#pragma unroll 1
            for (int b = b0; b < b0 + kPer; ++b) {
                const uint32_t d = tmem + ((uint32_t)(16 * (b >> 3)) << 16) + p * 256u + (uint32_t)(b & 7) * kTok;
                const uint64_t ad = smem_desc_sw128(s_base + F_OFF_W + b * 8192, 16, 1024);
                const uint64_t bd = smem_desc_sw128(s_base + F_OFF_A + b * 4096, 16, 1024);
#pragma unroll
                for (int s = 0; s < 4; ++s) umma_f16(d, ad + s * wstep, bd + s * 2, idesc, s > 0);   // K step of 16: 32 bytes of a swizzled row
            }
            umma_commit(bar_mma + 8 * p);
        }
        if (!ok) timed_out();
    }
    // teardown: the weight copy is the only thing that can still be in flight (after a wait ran out)
    if (tid == 32) mbar_wait(bar_w, 0);
    tc_fence_before();
    __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, 512);
}

// ---- gradients with respect to the weight blocks ------------------------------------------------------------------
//
//   D_b[m][a] = sum_t Z_b[t][m] * V_b[t][a]        for the 64 blocks b, contraction over ALL tokens
//
// V = x or the upstream gradient g, read as [t][a][b] with the block index b contiguous (exactly what pass 1 reads), and
// Z = the intermediate in the workspace layout [32-token tile][m / 16][t % 32][b][m % 16] that pass 1 writes:
//   dR[n2][k1][n1] = sum_t dv[t][n2][k1] x[t][n1][n2]:  V = x (b = n2, a = n1),  Z = pass 1 of (g, L^T) (m = k1)
//   dL[k1][k2][n2] = sum_t g[t][k2][k1] v[t][n2][k1]:   V = g (b = k1, a = k2),  Z = pass 1 of (x, R)   (m = n2), D = dL[k1]^T
// With the tokens as the K dimension both operands lie in shared memory as the forward passes already produce them: the swizzled
// tile [t][a] that pass 1 builds from 32-byte pieces of V is an MN-major operand (a row = one t), and a piece of the workspace,
// 16 values of m of one (t, b), is a row of a 32-byte-swizzled MN-major operand, so the copy engine brings Z as boxes
// [16 blocks][32 t][32 B].  Either may be the A operand: dL and dR leave as they are stored.
// A CTA owns 16 consecutive blocks and every (grid / 4)-th 32-token tile, accumulates its 16 [64 x 64] partial results in TMEM (M = 64:
// blocks 8 .. 15 at lane offset 16) and writes them once; a second kernel adds the shares in a fixed order.  Roles: warps 0..7 load V
// (the next tile's pieces are in flight while this one is multiplied), lane 0 of warp 8 copies Z (two buffers), lane 0 of warps 9 and
// 10 issue for 8 blocks each.  Bound, as the forward passes, by the requests for V's pieces (about 0.46 per cycle and SM).
// Measured, one B200, 5001 tokens: 26 us (37 for the kernel before it, which loaded, multiplied and waited in turn, 8 blocks at a time).
constexpr int G_OFF_V = 0;            // 16 operands [32 t][64 a] bf16, swizzled rows of 128 bytes                        65536
constexpr int G_OFF_Z = 65536;        // two buffers [m / 16][16 blocks][32 t][32 B]                                     131072
constexpr int G_OFF_BAR = 196608;     // bar_v, bar_mma[2], bar_z[2], tmem ptr, abort flag
constexpr int G_SMEM = G_OFF_BAR + 64;
constexpr int kGradLoadWarps = 8, kGradThreads = 32 * (kGradLoadWarps + 3);
constexpr int kGradShares = 37;       // 4 block groups x 37 = 148 CTAs
constexpr size_t kGradPartialBytes = (size_t)kGradShares * 64 * 4096 * 4;
static_assert(G_SMEM <= 232448, "shared-memory budget of the gradient kernel");

template <bool Z_IS_A>
__global__ void __launch_bounds__(kGradThreads, 1)
monarch64_wgrad_kernel(const __nv_bfloat16* __restrict__ in, const __grid_constant__ CUtensorMap map_z, float* __restrict__ partial,
                       long long T, int32_t* __restrict__ status) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t s_base = smem_u32(smem);
    const uint32_t bar_v = s_base + G_OFF_BAR, bar_mma = bar_v + 8, bar_z = bar_v + 24, s_tptr = bar_v + 40;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + G_OFF_BAR + 48);
    const int grp = blockIdx.x & 3, share = blockIdx.x >> 2, nshare = gridDim.x >> 2;
    const int ntiles = (int)((T + kTok - 1) / kTok);
    if (tid == 0) {
        mbar_init(bar_v, kGradLoadWarps);
        mbar_init(bar_mma, 2);         // both issuing threads; tile n uses barrier n % 2, so that a wait for tile n - 2 cannot miss it
        mbar_init(bar_mma + 8, 2);
        mbar_init(bar_z, 1);
        mbar_init(bar_z + 8, 1);
        *abort_flag = 0;
        fence_barrier_init();
        prefetch_tensormap(&map_z);
    }
    if (warp == 8) tmem_alloc(s_tptr, 512);
    // this CTA's quarter of a tile's lines of V, towards L2 as whole lines ahead of the pieces (see the forward passes)
    auto prefetch_tile = [&](int tile) {
        if (tile < ntiles) {
            const long long t0p = (long long)tile * kTok, rows = T - t0p >= kTok ? kTok : T - t0p;
            bulk_prefetch_l2(reinterpret_cast<const unsigned char*>(in) + t0p * 8192 + grp * (rows * 2048), (uint32_t)(rows * 2048));
        }
    };
    if (tid == 33) {
        prefetch_tile(share);
        prefetch_tile(share + nshare);
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the workspace was written by the kernel before this one
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + G_OFF_BAR + 40);
    bool ok = true;
    uint32_t n = 0;   // tiles begun
    if (warp < kGradLoadWarps) {
        const int t_in = tid >> 3, sub = tid & 7;   // (token, 8 consecutive a), as in pass 1
        uint32_t w[8][8];
        auto load_in = [&](int tile) {
            const long long t = (long long)tile * kTok + t_in;
            load_pieces<true>(w, reinterpret_cast<const unsigned char*>(in) + (size_t)t * 8192 + (size_t)(8 * sub) * 128 + grp * 32, t < T);
        };
        if (share < ntiles) load_in(share);
#pragma unroll 1
        for (int tile = share; tile < ntiles; tile += nshare, ++n) {
            if (__any_sync(~0u, *abort_flag != 0)) break;
            if (n > 0) ok = __all_sync(~0u, mbar_wait(bar_mma + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1));   // the UMMAs have read the operands
            if (!ok) break;
            store_pieces(w, smem + G_OFF_V + sw_off(t_in, sub));
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_v);
            if (tile + nshare < ntiles) load_in(tile + nshare);
            if (tid == 33) prefetch_tile(tile + 2 * nshare);
        }
        // the 16 accumulators: row r of block b sits in lane (r % 16) + 16 (b / 8) of lane quarter r / 16, columns 64 (b % 8) ..
        if (ok && n > 0) ok = __all_sync(~0u, mbar_wait(bar_mma + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1) && *abort_flag == 0);
        if (ok && n > 0) {
            tc_fence_after();
            const int q = warp & 3;
            const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16);
            // through the free operand buffers, 32 rows of 64 values per warp (pitch 68: no bank conflicts), so that whole rows leave
            float* st = reinterpret_cast<float*>(smem) + warp * (32 * 68);
#pragma unroll 1
            for (int cb = 4 * (warp >> 2); cb < 4 * (warp >> 2) + 4; ++cb) {
#pragma unroll 1
                for (int c0 = 0; c0 < 64; c0 += 32) {
                    float v[32];
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld8(t_lane + cb * 64 + c0 + 8 * c, v + 8 * c);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < 4; ++c) tmem_ld_fence8(v + 8 * c);
#pragma unroll
                    for (int c = 0; c < 32; c += 4)
                        *reinterpret_cast<float4*>(st + lane * 68 + c0 + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < 16; ++k) {   // row 2 k + lane / 16 of the 32: set row / 16, index row % 16 of this lane quarter
                    const int row = 2 * k + (lane >> 4);
                    float* dst = partial + (((size_t)share * 64 + grp * 16 + cb + 8 * (row >> 4)) * 64 + 16 * q + (row & 15)) * 64;
                    reinterpret_cast<float4*>(dst)[lane & 15] = *reinterpret_cast<const float4*>(st + row * 68 + 4 * (lane & 15));
                }
                __syncwarp();
            }
        }
    } else if (warp == 8) {
        if (lane == 0) {
            for (int tile = share; tile < ntiles && ok && *abort_flag == 0; tile += nshare, ++n) {
                const uint32_t z = s_base + G_OFF_Z + (n & 1) * 65536, bz = bar_z + 8 * (n & 1);
                if (n >= 2) ok = mbar_wait(bar_mma + 8 * (n & 1), ((n - 2) >> 1) & 1);   // the buffer's previous tile has been multiplied
                if (!ok) break;
                mbar_expect_tx(bz, 65536);
                for (int c = 0; c < 4; ++c) tma_load_3d(z + c * 16384, &map_z, 0, (tile * 4 + c) * kTok, 16 * grp, bz);
            }
            for (uint32_t i = n > 2 ? n - 2 : 0; i < n; ++i) mbar_wait(bar_z + 8 * (i & 1), (i >> 1) & 1);   // nothing is left in flight
        }
    } else if (elect_one()) {
        const uint32_t idesc = instr_desc_bf16(64, 64, true, true);
        const int b0 = (warp - 9) * 8;
        for (int tile = share; tile < ntiles && ok && *abort_flag == 0; tile += nshare, ++n) {
            ok = mbar_wait(bar_v, n & 1) && mbar_wait(bar_z + 8 * (n & 1), (n >> 1) & 1);
            if (!ok) break;
            tc_fence_after();
            const uint32_t z = s_base + G_OFF_Z + (n & 1) * 65536;
#pragma unroll 1
            for (int b = b0; b < b0 + 8; ++b) {
                const uint32_t d = tmem + ((uint32_t)(16 * (b >> 3)) << 16) + (uint32_t)(b & 7) * 64;
                const uint64_t zd = smem_desc_sw32(z + b * 1024, 16384, 256), vd = smem_desc_sw128(s_base + G_OFF_V + b * 4096, 8192, 1024);
#pragma unroll
                for (int k = 0; k < 2; ++k)   // 16 tokens per instruction
                    umma_f16(d, Z_IS_A ? zd + k * 32 : vd + k * 128, Z_IS_A ? vd + k * 128 : zd + k * 32, idesc, (n > 0 || k > 0) ? 1u : 0u);
            }
            umma_commit(bar_mma + 8 * (n & 1));
        }
    }
    if (!ok) {
        atomicExch(status, (int32_t)M2_ERR_TIMEOUT);
        *abort_flag = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 8) tmem_dealloc(tmem, 512);
}

// out = the sum of the shares, four values per thread (nshare = 0: zeros): warp y of a block adds the shares y, y + 8, .. in order, the
// eight sums are added in order.  Bound by the shares' bytes (39 MB for 37 shares) once a warp's loads are in flight together: one thread per
// value walking all shares 11.1 us, warps whose last loads came one by one 10.1, now 8.4 (cold); [5001] tokens forward and backward 166.6 -> 165.4.
__global__ void __launch_bounds__(256) wgrad_reduce_kernel(const float4* __restrict__ partial, float4* __restrict__ out, int nshare) {
    __shared__ float4 part[8][32];
    const int lane = threadIdx.x & 31, y = threadIdx.x >> 5, e = blockIdx.x * 32 + lane;   // < 64 * 4096 / 4
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = y; s0 < nshare; s0 += 40) {
        float4 v[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) v[q] = s0 + 8 * q < nshare ? __ldcg(partial + (size_t)(s0 + 8 * q) * 65536 + e) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            acc.x += v[q].x;
            acc.y += v[q].y;
            acc.z += v[q].z;
            acc.w += v[q].w;
        }
    }
    part[y][lane] = acc;
    __syncthreads();
    if (y == 0) {
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            const float4 v = part[q][lane];
            acc.x += v.x;
            acc.y += v.y;
            acc.z += v.z;
            acc.w += v.w;
        }
        out[e] = acc;
    }
}

int64_t wgrad_workspace_bytes(const m2_plan* pl, int64_t T) { return covered(pl) ? workspace_bytes(pl, T) + (int64_t)kGradPartialBytes : 0; }

static cudaLaunchConfig_t early_launch(unsigned grid, int threads, size_t smem, cudaStream_t stream, cudaLaunchAttribute* attr) {
    attr->id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr->val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}
static unsigned fwd_grid(int64_t T) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long nitems = 4 * ((T + kTok - 1) / kTok);
    const long long ctas = (sms / 4) * 4 > 4 ? (sms / 4) * 4 : 4;   // a multiple of 4: a CTA keeps its block group
    return (unsigned)(nitems < ctas ? nitems : ctas);
}
// weight blocks as TMA tiles: [64 blocks x 64 rows][64] bf16, one box = one block, 128-byte swizzle
static bool weight_map(CUtensorMap* m, const void* W) {
    const cuuint64_t gdim[2] = {64, 64 * 64}, gstr[1] = {128};
    const cuuint32_t box[2] = {64, 64};
    return tma_host::encode_sw128_bf16(m, W, 2, gdim, gstr, box);
}

int32_t wgrad(const m2_plan* pl, const void* X, const void* G, const void* L, const void* R, float* dL, float* dR, int64_t T, void* ws,
              cudaStream_t stream) {
    if (!covered(pl)) return M2_ERR_UNSUPPORTED;
    unsigned char* zws = static_cast<unsigned char*>(ws);
    float* partial = reinterpret_cast<float*>(zws + workspace_bytes(pl, T));
    const int64_t ntiles = (T + kTok - 1) / kTok;
    unsigned shares = fwd_grid(T) / 4;
    if (shares > kGradShares) shares = kGradShares;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t red = early_launch(2048, 256, 0, stream, &attr);
    if (T == 0) {
        if (cudaLaunchKernelEx(&red, wgrad_reduce_kernel, (const float4*)partial, (float4*)dL, 0) != cudaSuccess ||
            cudaLaunchKernelEx(&red, wgrad_reduce_kernel, (const float4*)partial, (float4*)dR, 0) != cudaSuccess)
            return M2_ERR_CUDA;
        pl->launches += 2;
        return M2_OK;
    }
    if (ntiles > 0x1000000) return M2_ERR_UNSUPPORTED;   // (row index of the workspace map)
    // the workspace as (16 values of m | (tile, m / 16, t), 2 KB apart | block, 32 B apart): a box lands block by block
    alignas(64) CUtensorMap mr, ml, mz;
    const cuuint64_t zdim[3] = {16, (cuuint64_t)ntiles * 4 * kTok, 64}, zstr[2] = {2048, 32};
    const cuuint32_t zbox[3] = {16, (cuuint32_t)kTok, 16};
    if (!weight_map(&mr, R) || !weight_map(&ml, L) || !tma_host::encode_sw32_bf16(&mz, zws, 3, zdim, zstr, zbox)) return M2_ERR_UNSUPPORTED;
    const cudaLaunchConfig_t p1 = early_launch(fwd_grid(T), kFwdThreads, F_SMEM_BYTES, stream, &attr);
    const cudaLaunchConfig_t wg = early_launch(4 * shares, kGradThreads, G_SMEM, stream, &attr);
    const __nv_bfloat16 *x = (const __nv_bfloat16*)X, *g = (const __nv_bfloat16*)G, *none = nullptr;
    __nv_bfloat16* z = (__nv_bfloat16*)zws;
    // dL: v = R-stage of x, then sum_t g (x) v per block k1;  dR: dv = L^T-stage of g, then sum_t dv (x) x per block n2
    auto first = (reinterpret_cast<uintptr_t>(X) & 31u) == 0 ? monarch64_fwd_kernel<1, false> : monarch64_fwd_kernel<1, true>;
    if (cudaLaunchKernelEx(&p1, first, x, mr, mr, z, (long long)T, pl->d_status, none, 1LL, 0, 0, 0) != cudaSuccess ||
        cudaLaunchKernelEx(&wg, monarch64_wgrad_kernel<false>, g, mz, partial, (long long)T, pl->d_status) != cudaSuccess ||
        cudaLaunchKernelEx(&red, wgrad_reduce_kernel, (const float4*)partial, (float4*)dL, (int)shares) != cudaSuccess ||
        cudaLaunchKernelEx(&p1, monarch64_fwd_kernel<1, true>, g, ml, ml, z, (long long)T, pl->d_status, none, 1LL, 0, 0, 1) != cudaSuccess ||
        cudaLaunchKernelEx(&wg, monarch64_wgrad_kernel<true>, x, mz, partial, (long long)T, pl->d_status) != cudaSuccess ||
        cudaLaunchKernelEx(&red, wgrad_reduce_kernel, (const float4*)partial, (float4*)dR, (int)shares) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->last_kernel = "matmul_wgrad_umma_64x64";
    pl->launches += 6;
    return M2_OK;
}

bool covered(const m2_plan* pl) { return pl->dtype == M2_BF16 && pl->p == 2 && pl->dims[0] == 64 && pl->dims[1] == 64; }

// whole token tiles: the last tile's slab is written in full
int64_t workspace_bytes(const m2_plan* pl, int64_t T) { return covered(pl) ? ((T + kTileT - 1) / kTileT) * kTileT * 4096 * 2 : 0; }

cudaError_t prepare(const m2_plan* pl) {
    if (!covered(pl)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(monarch64_pass_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_pass_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_wgrad_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_wgrad_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_fwd_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_fwd_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_fwd_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(monarch64_fwd_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES);
    return e;
}

// 128 tokens x 8 blocks per CTA (16-byte pieces): serves inputs that are only 16-byte aligned
static int32_t matmul_g8(const m2_plan* pl, const void* X, const void* L, const void* R, void* Y, int64_t T, void* ws, const void* Kmul,
               int64_t Hk, int relu, cudaStream_t stream) {
    if (!covered(pl)) return M2_ERR_UNSUPPORTED;
    if (T == 0) return M2_OK;
    dim3 grid(8, (unsigned)((T + kTileT - 1) / kTileT));
    // y[t][k2][k1] seen as (k1 64 | t, stride 8 KB | k2, stride 128 B); box = 8 k1 x 128 tokens x 64 k2
    alignas(64) CUtensorMap my;
    const cuuint64_t gdim[3] = {64, (cuuint64_t)T, 64}, gstr[2] = {8192, 128};
    const cuuint32_t box[3] = {8, (cuuint32_t)kTileT, 64};
    if (!tma_host::encode_bf16(&my, Y, 3, gdim, gstr, box)) return M2_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, monarch64_pass_kernel<1>, (const __nv_bfloat16*)X, (const __nv_bfloat16*)R, my, (__nv_bfloat16*)ws,
                           (long long)T, pl->d_status, (const __nv_bfloat16*)nullptr, 1LL, 0) != cudaSuccess)
        return M2_ERR_CUDA;
    if (cudaLaunchKernelEx(&cfg, monarch64_pass_kernel<2>, (const __nv_bfloat16*)ws, (const __nv_bfloat16*)L, my,
                           (__nv_bfloat16*)nullptr, (long long)T, pl->d_status, (const __nv_bfloat16*)Kmul, (long long)(Hk > 0 ? Hk : 1),
                           relu) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->last_kernel = "matmul_umma_64x64_g8";
    pl->launches += 2;
    return M2_OK;
}

static int32_t matmul_impl(const m2_plan* pl, const void* X, const void* L, const void* R, void* Y, int64_t T, void* ws, const void* Kmul,
                           int64_t Hk, int relu, int selftest, int wt, cudaStream_t stream) {
    if (!covered(pl)) return M2_ERR_UNSUPPORTED;
    if (T == 0) return selftest ? M2_ERR_UNSUPPORTED : M2_OK;
    // the loads of pass 1 want x on a 32-byte boundary (torch allocations are; a view need not be)
    if ((reinterpret_cast<uintptr_t>(X) & 31u) != 0)
        return selftest || wt ? M2_ERR_UNSUPPORTED : matmul_g8(pl, X, L, R, Y, T, ws, Kmul, Hk, relu, stream);
    alignas(64) CUtensorMap mr, ml, my;
    if (!weight_map(&mr, R) || !weight_map(&ml, L)) return M2_ERR_UNSUPPORTED;
    // y[t][k2][k1] seen as (k1 64 | k2, stride 128 B | t, stride 8 KB); box = 16 k1 x 16 k2 x 4 tokens, 32-byte swizzle
    const cuuint64_t ydim[3] = {64, 64, (cuuint64_t)T}, ystr[2] = {128, 8192};
    const cuuint32_t ybox[3] = {16, 16, 4};
    if (!tma_host::encode_sw32_bf16(&my, Y, 3, ydim, ystr, ybox)) return M2_ERR_UNSUPPORTED;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = early_launch(fwd_grid(T), kFwdThreads, F_SMEM_BYTES, stream, &attr);
    if (cudaLaunchKernelEx(&cfg, wt ? monarch64_fwd_kernel<1, true> : monarch64_fwd_kernel<1, false>, (const __nv_bfloat16*)X, mr, my, (__nv_bfloat16*)ws, (long long)T, pl->d_status,
                           (const __nv_bfloat16*)nullptr, 1LL, 0, selftest, wt) != cudaSuccess)
        return M2_ERR_CUDA;
    if (cudaLaunchKernelEx(&cfg, wt ? monarch64_fwd_kernel<2, true> : monarch64_fwd_kernel<2, false>, (const __nv_bfloat16*)ws, ml, my, (__nv_bfloat16*)Y, (long long)T, pl->d_status,
                           (const __nv_bfloat16*)Kmul, (long long)(Hk > 0 ? Hk : 1), relu, selftest, wt) != cudaSuccess)
        return M2_ERR_CUDA;
    pl->last_kernel = "matmul_umma_64x64";
    pl->launches += 2;
    return M2_OK;
}

int32_t matmul(const m2_plan* pl, const void* X, const void* L, const void* R, void* Y, int64_t T, void* ws, const void* Kmul,
               int64_t Hk, int relu, cudaStream_t stream) {
    return matmul_impl(pl, X, L, R, Y, T, ws, Kmul, Hk, relu, 0, 0, stream);
}

int32_t matmul_bwd_input(const m2_plan* pl, const void* G, const void* L, const void* R, void* dX, int64_t T, void* ws, cudaStream_t stream) {
    return matmul_impl(pl, G, R, L, dX, T, ws, nullptr, 1, 0, 0, 1, stream);   // M^T: the factors in the opposite order, blocks transposed
}

int32_t matmul_wait_selftest(const m2_plan* pl, const void* X, const void* L, const void* R, void* Y, int64_t T, void* ws,
                             cudaStream_t stream) {
    return matmul_impl(pl, X, L, R, Y, T, ws, nullptr, 1, 0, 1, 0, stream);
}

}  // namespace m2mm
