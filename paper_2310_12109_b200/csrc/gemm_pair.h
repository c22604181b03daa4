// Batched GEMM on CTA pairs (internal header).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "m2_plan.h"

namespace m2c {

// bf16 tensor p[bt][j][i1][i0]: extents n0 (contiguous), n1, nj, nbt; strides in elements, multiples of 8
struct PairTensor {
    const void* p;
    int64_t n0, n1, s1, nj, sj, nbt, sbt;
};
// O[w][bt][j][rows][cols] = A[w] B, contracted over k (a multiple of 64).  A: K-major (n0 = k, n1 = row) or M-major (n0 = row, n1 = k);
// B: N-major (n0 = column, n1 = k) or K-major (n0 = k, n1 = column); O: n0 = column, n1 = row.  One operand carries the batch index.
struct PairGemm {
    int weights = 1;             // 1 .. 3 weights A against the same B, one output each
    PairTensor a[3], b, o[3];
    int64_t rows = 0, cols = 0, k = 0;
    int a_mmajor = 0, b_kmajor = 0, a_batched = 0;
    PairTensor kmul = {};        // factor on the result, shared by the batch: n0 = column, n1 = row; p == nullptr: none
    int relu = 0;                // after the factor
};
int32_t gemm_pair(const m2_plan* pl, const PairGemm& g, cudaStream_t stream);

}  // namespace m2c
