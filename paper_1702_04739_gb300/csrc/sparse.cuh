// sparse.cuh -- the rows of one set by their non-zeros.
#pragma once
#include "common.cuh"
#include "dwmath.cuh"

namespace iso {

// Row r: dimensions rcol and values rval of entries rowptr[r] .. rowptr[r + 1],
// ascending; the first `width` of them also in ell, slot by slot over the 32
// rows of a group (value, dimension as bits), so that 32 threads with a row
// each read whole lines.  Group g (rows 32 g .. + 31): its entries by dimension,
// then row, in gent (value, row of the group's 32 as bits) at rowptr[32 g] + the
// offset o >> 6, o & 63 of them, o = goff of (g, t): the four groups of a tile
// of 128 rows side by side.
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
    float *root = nullptr;             // |x|, rounded up
    int32_t width = 0;
    float2 *ell = nullptr;             // [n_pad / 32][width][32]

    __device__ const uint32_t *table(int64_t g) const { return goff + (g >> 2) * d * 4 + (g & 3); }     // + 4 t
    __device__ const float2 *slots(int64_t r) const { return ell + (r >> 5) * width * 32 + (r & 31); }  // + 32 k

    void carve(Arena &A, int64_t n, int32_t d, int64_t nnz);
};

// Non-zeros and the largest |x|^2 of the rows of X into stat[0..1] (64 bits)
// and [2] (FP32 bits), zeroed before.
cudaError_t sparse_stats(const float *X, int64_t n, int32_t d, uint32_t *stat, cudaStream_t s);
// Whether rows of that many non-zeros take the sparse kernels.
bool sparse_pays(int64_t n, int32_t d, int64_t nnz, float norm_max);
// Calls f(value of j, entry of the group) for every dimension that row j and a
// row of group g both hold.  Each look-up is two reads that wait for one
// another (the table, the entries): the next four's table entries are on their
// way, and four entries of two look-ups each are read at a time (rows in a
// clustered order share dimensions: five entries a look-up at 50,000 x 4,096).
template <class F>
__device__ __forceinline__ void sparse_products(const SparseRows &R, int64_t j, int64_t g, F f) {
    const int32_t e0 = R.rowptr[j], e1 = R.rowptr[j + 1];
    const int32_t len = e1 - e0 < R.width ? e1 - e0 : R.width;
    const uint32_t *go = R.table(g);
    const float2 *sl = R.slots(j), *ge = R.gent + R.rowptr[32 * g];
    auto fetch = [&](int32_t k, uint32_t (&o)[4], float (&v)[4]) {
        float2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k + u < len) x[u] = sl[(int64_t)(k + u) * 32];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            o[u] = 0u;
            v[u] = 0.f;
            if (k + u < len) {
                o[u] = go[(int64_t)__float_as_int(x[u].y) * 4];
                v[u] = x[u].x;
            }
        }
    };
    uint32_t o[4], on[4];
    float v[4], vn[4];
    fetch(0, o, v);
    for (int32_t k = 0; k < len; k += 4) {
        fetch(k + 4, on, vn);
#pragma unroll
        for (int u = 0; u < 4; u += 2) {
            const int c0 = (int)(o[u] & 63u), c1 = (int)(o[u + 1] & 63u);
            const float2 *g0 = ge + (o[u] >> 6), *g1 = ge + (o[u + 1] >> 6);
            for (int q = 0; q < c0 || q < c1; q += 4) {
                float2 x[4], y[4];
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    if (q + z < c0) x[z] = g0[q + z];
                    if (q + z < c1) y[z] = g1[q + z];
                }
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                    if (q + z < c0) f(v[u], x[z]);
                    if (q + z < c1) f(v[u + 1], y[z]);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            o[u] = on[u];
            v[u] = vn[u];
        }
    }
    for (int32_t e = e0 + len; e < e1; ++e) {
        const uint32_t t = go[(int64_t)R.rcol[e] * 4];
        for (int q = 0; q < (int)(t & 63u); ++q) f(R.rval[e], ge[(t >> 6) + q]);
    }
}

// Squared distance of rows i and j as a double-word, along the two lists (a
// dimension that neither holds adds nothing).  Four squares are summed before
// they join the sum, as in the dense direct sums.
__device__ __forceinline__ void sparse_dist2(const SparseRows &R, int64_t i, int64_t j, float &h, float &l) {
    int32_t a = R.rowptr[i], b = R.rowptr[j];
    const int32_t ea = R.rowptr[i + 1], eb = R.rowptr[j + 1];
    float fh = 0.f, fl = 0.f;
    h = l = 0.f;
    for (int c = 1; a < ea || b < eb; ++c) {
        const int32_t ta = a < ea ? R.rcol[a] : INT32_MAX, tb = b < eb ? R.rcol[b] : INT32_MAX;
        const float x = ta <= tb ? R.rval[a++] : 0.f, y = tb <= ta ? R.rval[b++] : 0.f;
        float p, q;
        dw_square_diff(x, y, p, q);
        dw_add(fh, fl, p, q);
        if ((c & 3) == 0) {
            dw_add(h, l, fh, fl);
            fh = fl = 0.f;
        }
    }
    dw_add(h, l, fh, fl);
}

constexpr int32_t SPARSE_MIN_D = 512, SPARSE_MAX_D = 16384;
cudaError_t sparse_build(SparseRows &R, const float *X, cudaStream_t s);
// FP32 squared distances of all pairs (ld words a row), the sign set where the
// Gram's roundings would have passed 3 % and the distance is a direct sum,
// rounded once
cudaError_t sparse_dist(const SparseRows &R, float *D, int64_t ld, cudaStream_t s);

}  // namespace iso
