// Short causal convolutions (bf16, n <= 256) as Toeplitz products: y[b][t] = sum_s k[t - s] x[b][s] per channel.
//
// For n this short the n^2 / 2 products per row, done by matrix instructions, cost less than a transform of 2 n points goes through in
// hand-offs and padding: x is read once, y written once, nothing else moves.  M = 16 batch rows, N = 8 positions t, K = 16 positions s;
// a tile of the Toeplitz factor depends on t - s only, so its fragment for distance d (in steps of 8) is one word per lane of a table
// P[u] = (k[u], k[u - 1]), the second half of one fragment is the first half of the next, and a warp that walks s re-reads nothing.
// The kernel is fp32: its values are split into two bf16 parts (16 bits of mantissa) and both are multiplied; the result's distance from
// the exact sum is the rounding of the output, 1.65e-3 to 1.68e-3 for N(0, 1) rows of 37 to 256 positions as with fp32 transforms (the
// bf16 transforms of the 32 x 16 plan: 3.2e-3).  Lags below zero exist when the spectrum was conjugated (the
// transposed convolution); a direction without a non-zero value is not walked.
//
// An item is one channel and 32 (16) batch rows; a warp takes 32 positions (with 16 the operand fragments' way from shared memory was
// as long as the multiplication).  The blocks are persistent: the
// next item's rows (cp.async, second buffer) and kernel values (registers) are on their way while the current one is multiplied.  An item
// of n = 256 is 1152 matrix instructions, of which an SM takes 0.47 a cycle; the three sets below keep that pipe 57 % busy (issue slots
// 42 %, load/store data pipe 45 %, 20 warps per SM): the rest is the fragments' latency between two barriers per item and a last round
// of 2304 items on 444 blocks that is a fifth full.
// Measured, one B200: bf16 [32][768][256] 15.8 us (20.2 with 512-point transforms on the tensor cores), [32][768][200] 13.5 us, the three
// short convolutions of the Hyena layer at [32][768][256] in one launch 43 us (3 x 23.5).  Of these sizes, the ones with full items are
// toeplitz_umma.cu's now (11.9, 11.8 and 28 us; umma_pays has the line): this kernel runs shorter rows, odd lengths, small batches, few items.
#include "m2_plan.h"
#include "mma_sync.cuh"
#include "toeplitz_mma.h"

namespace m2t {

constexpr int kThreads = 256, kWarps = kThreads / 32, kBlocksPerSm = 3;

__host__ __device__ constexpr int padded(int n) { return (n + 15) / 16 * 16; }
__host__ __device__ constexpr int pitch(int n) { return padded(n) + 8; }   // bf16 elements: rows 16 bytes apart mod 128
__host__ __device__ constexpr int table(int n) { return 2 * padded(n) + 32; }   // entries; the last ones are zero (a half-empty last tile)
__host__ __device__ constexpr int smem_bytes(int n, int rows) { return 2 * rows * pitch(n) * 2 + 2 * table(n) * 4; }
static_assert(2 * kMaxN <= 2 * kThreads && kMaxN <= 32 * kWarps, "two table entries per thread, one tile per warp");

struct Sets {
    Rows r[3];
};

template <int MT>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    toeplitz_kernel(const Sets sets, int items, int B, int H, int n, int N, int kf_group) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kRows = 16 * MT, kR = kRows / kWarps;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int np = padded(n), ld = pitch(n);
    __nv_bfloat16* xbuf = reinterpret_cast<__nv_bfloat16*>(smem);   // two buffers [kRows][ld]
    uint32_t* ph = reinterpret_cast<uint32_t*>(xbuf + 2 * kRows * ld);   // P[u] at u + np, upper parts
    uint32_t* pl = ph + table(n);                                         // lower parts
    const int m8 = lane >> 3, r8 = lane & 7, g = lane >> 2, c2 = 2 * (lane & 3);
    const int tiles = np / 16, wide = (tiles + 1) / 2;
    if (tid < 32) ph[2 * np + tid] = pl[2 * np + tid] = 0u;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    float ka[2], kb[2];   // this thread's entries of the next table: lags u and u - 1
    // items in the order set, batch chunk, channel; stepping from one to the next takes no division
    struct Item {
        int set, b0, h;
    };
    auto advance = [&](Item& v, int by) {
        v.h += by;
        while (v.h >= H) {
            v.h -= H;
            v.b0 += kRows;
            if (v.b0 >= B) {
                v.b0 = 0;
                ++v.set;
            }
        }
    };
    auto fetch = [&](const Item& v, int buf) {
        const int h = v.h, b0 = v.b0;
        const __nv_bfloat16* x = static_cast<const __nv_bfloat16*>(v.set == 0 ? sets.r[0].x : v.set == 1 ? sets.r[1].x : sets.r[2].x);
        const float* kt = (v.set == 0 ? sets.r[0].kt : v.set == 1 ? sets.r[1].kt : sets.r[2].kt) + (size_t)(kf_group == 1 ? h : h / kf_group) * N;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int u = tid + q * kThreads - np;   // (entries past 2 np are not stored)
            ka[q] = u > -n && u < n ? __ldg(kt + (u & (N - 1))) : 0.f;
            kb[q] = u - 1 > -n && u - 1 < n ? __ldg(kt + ((u - 1) & (N - 1))) : 0.f;
        }
        __nv_bfloat16* xs = xbuf + buf * kRows * ld;
        if (n % 8 == 0) {   // 16-byte pieces never straddle a row
            for (int c = lane * 8; c < np; c += 256)
#pragma unroll
                for (int q = 0; q < kR; ++q) {
                    const int r = warp + kWarps * q, b = b0 + r;
                    const bool in = b < B && c < n;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(xs + r * ld + c)),
                                 "l"(x + (in ? ((size_t)b * H + h) * n + c : 0)), "r"(in ? 16 : 0)
                                 : "memory");
                }
        } else if (n % 2 == 0) {
            for (int c = lane * 2; c < np; c += 64)
#pragma unroll
                for (int q = 0; q < kR; ++q) {
                    const int r = warp + kWarps * q, b = b0 + r;
                    const bool in = b < B && c < n;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_addr(xs + r * ld + c)),
                                 "l"(x + (in ? ((size_t)b * H + h) * n + c : 0)), "r"(in ? 4 : 0)
                                 : "memory");
                }
        } else {
            for (int r = warp; r < kRows; r += kWarps)
                for (int c = lane; c < np; c += 32)
                    xs[r * ld + c] = b0 + r < B && c < n ? x[((size_t)(b0 + r) * H + h) * n + c] : __float2bfloat16_rn(0.f);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    int buf = 0;
    Item cur = {0, 0, 0};
    advance(cur, blockIdx.x);
    if ((int)blockIdx.x < items) fetch(cur, 0);
    for (int it = blockIdx.x; it < items; it += gridDim.x, buf ^= 1) {
        bool later = false, earlier = false;   // non-zero lags on either side
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = tid + q * kThreads, u = i - np;
            if (i < 2 * np) {
                later = later || (u > 0 && ka[q] != 0.f);
                earlier = earlier || (u < 0 && ka[q] != 0.f);
                const uint32_t w = bf2(ka[q], kb[q]);
                ph[i] = w;
                pl[i] = bf2(ka[q] - __uint_as_float(w << 16), kb[q] - __uint_as_float(w & 0xffff0000u));
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        later = __syncthreads_or(later);
        earlier = __syncthreads_or(earlier);
        const int h = cur.h, b0 = cur.b0;
        __nv_bfloat16* y = static_cast<__nv_bfloat16*>(cur.set == 0 ? sets.r[0].y : cur.set == 1 ? sets.r[1].y : sets.r[2].y);
        advance(cur, gridDim.x);
        if (it + (int)gridDim.x < items) fetch(cur, buf ^ 1);
        const uint32_t ax = smem_addr(xbuf + buf * kRows * ld + ((m8 & 1) * 8 + r8) * ld + (m8 >> 1) * 8);
        // tiles of 32 positions, one per warp; warps w and w + 4, on one scheduler, get a short and a long one
        const int half = (wide + 1) / 2, tj = warp < 4 ? warp : wide - 1 - (warp - 4);
        if (warp < 4 ? warp < half : warp - 4 < wide - half) {
            const int s0 = later ? 0 : 2 * tj, s1 = earlier || 2 * tj + 1 > tiles - 1 ? tiles - 1 : 2 * tj + 1;
            float o[MT][4][4] = {};
            const uint32_t* qh = ph + np + g - c2 + 32 * tj - 16 * s0;
            const uint32_t* ql = pl + np + g - c2 + 32 * tj - 16 * s0;
            uint32_t wh[5], wl[5];   // the fragments' words at distances -1 .. 3
#pragma unroll
            for (int e = 2; e < 5; ++e) {
                wh[e] = qh[8 * (e - 1)];
                wl[e] = ql[8 * (e - 1)];
            }
#pragma unroll 2
            for (int si = s0; si <= s1; ++si, qh -= 16, ql -= 16) {
                wh[1] = qh[0];
                wh[0] = qh[-8];
                wl[1] = ql[0];
                wl[0] = ql[-8];
                uint32_t fa[MT][4];
#pragma unroll
                for (int m = 0; m < MT; ++m) ldsm4(fa[m], ax + m * 32 * ld + si * 32);
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int e = 0; e < 4; ++e) mma(o[m][e], fa[m], wh[e + 1], wh[e]);
#pragma unroll
                for (int m = 0; m < MT; ++m)
#pragma unroll
                    for (int e = 0; e < 4; ++e) mma(o[m][e], fa[m], wl[e + 1], wl[e]);
#pragma unroll
                for (int e = 4; e >= 2; --e) {
                    wh[e] = wh[e - 2];
                    wl[e] = wl[e - 2];
                }
            }
            // a lane holds two positions of rows g and g + 8; the other half of a 32-byte sector comes with the neighbouring e
            const int t0 = tj * 32 + c2;
            const size_t rstep = (size_t)8 * H * n;
            __nv_bfloat16* d = y + ((size_t)(b0 + g) * H + h) * n + t0;
#pragma unroll
            for (int q = 0; q < 2 * MT; ++q, d += rstep) {
                if (b0 + g + 8 * q >= B) break;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t w = bf2(o[q / 2][e][2 * (q & 1)], o[q / 2][e][2 * (q & 1) + 1]);
                    if (n % 2 == 0) {
                        if (t0 + 8 * e < n) *reinterpret_cast<uint32_t*>(d + 8 * e) = w;
                    } else {
                        if (t0 + 8 * e < n) reinterpret_cast<unsigned short*>(d)[8 * e] = (unsigned short)w;
                        if (t0 + 8 * e + 1 < n) reinterpret_cast<unsigned short*>(d)[8 * e + 1] = (unsigned short)(w >> 16);
                    }
                }
            }
        }
        __syncthreads();   // the table and this buffer are free
    }
}

bool has_time_kernel(const m2_plan* pl) { return pl->dtype == M2_BF16 && pl->d_fft != nullptr && pl->N >= 256 && pl->N <= 512; }

const float* time_kernel(const m2_plan* pl, const void* kf, int64_t H) {
    const int64_t orders = pl->N == 512 && pl->umma != nullptr ? 2 : 1;   // (the tensor-core order of the 32 x 16 plan lies in between)
    return reinterpret_cast<const float*>(static_cast<const unsigned char*>(kf) + orders * H * pl->N * 8);
}

int32_t conv(const m2_plan* pl, const Rows* sets, int count, int64_t B, int64_t H, int64_t n, int kf_group, cudaStream_t stream) {
    if (!has_time_kernel(pl) || n > kMaxN || 2 * n > pl->N || count < 1 || count > 3) return M2_ERR_UNSUPPORTED;
    if (umma_pays(pl, count, B, H, n)) {
        const int32_t rc = conv_umma(pl, sets, count, B, H, n, kf_group, stream);
        if (rc != M2_ERR_UNSUPPORTED) return rc;
    }
    Sets s;
    for (int i = 0; i < 3; ++i) s.r[i] = sets[i < count ? i : 0];
    const int rows = B <= 16 ? 16 : 32;
    const int64_t per_set = H * ((B + rows - 1) / rows), items = per_set * count;
    if (items == 0) return M2_OK;
    if (items > 0x3fffffffLL) return M2_ERR_UNSUPPORTED;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t most = (int64_t)sms * kBlocksPerSm;
    auto kern = rows == 16 ? toeplitz_kernel<1> : toeplitz_kernel<2>;
    const int smem = smem_bytes((int)n, rows);
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(kMaxN, rows)) != cudaSuccess)
        return M2_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items < most ? items : most));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, s, (int)items, (int)B, (int)H, (int)n, (int)pl->N, kf_group) != cudaSuccess) return M2_ERR_CUDA;
    pl->last_kernel = "conv_toeplitz_mma";
    pl->launches += 1;
    return M2_OK;
}

}  // namespace m2t
