// sparse.cuh -- the rows of one set by their non-zeros.
#pragma once
#include "common.cuh"

namespace iso {

// Row r: dimensions rcol and values rval of entries rowptr[r] .. rowptr[r + 1],
// ascending.  Group g (rows 32 g .. + 31): its entries by dimension, then row,
// in gent (value, row of the group's 32 as bits) at rowptr[32 g] + the offset
// goff[g d + t] >> 6, goff & 63 of them.
struct SparseRows {
    int64_t n = 0, n_pad = 0;          // rows; rounded up to whole tiles of 128 (no entries)
    int32_t d = 0;
    int64_t cap = 0;                   // entries the arrays hold
    int32_t *rowptr = nullptr, *cnt = nullptr, *tmp = nullptr;
    int32_t *rcol = nullptr;
    float *rval = nullptr;
    uint32_t *goff = nullptr;
    float2 *gent = nullptr;
    float2 *norm = nullptr;            // |x|^2 as a double-word

    void carve(Arena &A, int64_t n, int32_t d, int64_t nnz);
};

// Non-zeros, the longest row and the largest |x|^2 of the rows of X into
// stat[0..1] (64 bits), [2] and [3] (FP32 bits), zeroed before.
cudaError_t sparse_stats(const float *X, int64_t n, int32_t d, uint32_t *stat, cudaStream_t s);
// Whether rows of that many non-zeros take the sparse kernels.
bool sparse_pays(int64_t n, int32_t d, int64_t nnz, float norm_max);
constexpr int32_t SPARSE_MIN_D = 512, SPARSE_MAX_D = 16384;
cudaError_t sparse_build(SparseRows &R, const float *X, cudaStream_t s);
// FP32 squared distances of all pairs (ld words a row)
cudaError_t sparse_dist(const SparseRows &R, float *D, int64_t ld, cudaStream_t s);

}  // namespace iso
