// sparse.cu -- rows with few non-zeros: their lists, and all pairs' squared
// distances from them.
//
// A pair's product needs the dimensions both rows hold: at 50,000 x 4,096
// with 41 non-zeros a row about one per pair, where the dense kernels run
// through all 4,096.  The Gram of 128 rows and 64 columns goes by look-ups: a
// thread has one column and 32 rows, walks the column's non-zeros and finds
// the rows that hold each dimension in the rows' table (goff), whose entries
// it multiplies into its own 32 sums in shared memory.  Every sum has one
// owner and a fixed order.  Bound by the latency of the look-ups: all pairs of
// 20,000 x 4,096 took 3.1 ms with the columns' lists read row by row and one
// look-up at a time, 1.2 slot by slot and four at a time.
#include <math.h>

#include "sparse.cuh"

namespace iso {
namespace {
__global__ void __launch_bounds__(256) k_sp_stats(const float *__restrict__ X, int64_t n, int32_t d,
                                                  uint32_t *__restrict__ stat) {
    const int lane = threadIdx.x & 31;
    unsigned long long total = 0;
    float nmax = 0.0f;
    const int64_t gs = (int64_t)gridDim.x * 8;
    for (int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); r < n; r += gs) {
        unsigned c = 0;
        float q = 0.0f;
        for (int t = lane; t < d; t += 32) {
            const float v = X[r * d + t];
            c += v != 0.0f;
            q = fmaf(v, v, q);
        }
        for (int o = 16; o > 0; o >>= 1) {
            c += __shfl_xor_sync(0xffffffffu, c, o);
            q += __shfl_xor_sync(0xffffffffu, q, o);
        }
        total += c;
        nmax = fmaxf(nmax, q);
    }
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(stat), total);
        atomicMax(stat + 2, __float_as_uint(nmax));          // (non-negative floats: their bits are in order)
    }
}

// one warp per padded row: its non-zeros, |x|^2 (FP64 sum) as a double-word, |x|
// rounded up
__global__ void __launch_bounds__(256) k_sp_count(const float *__restrict__ X, int64_t n, int64_t n_pad, int32_t d,
                                                  int32_t *__restrict__ cnt, float2 *__restrict__ norm, float *__restrict__ root) {
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r > n_pad) return;
    int c = 0;
    double q = 0.0;
    if (r < n)
        for (int t = lane; t < d; t += 32) {
            const float v = X[r * d + t];
            c += v != 0.0f;
            q = fma((double)v, (double)v, q);
        }
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if (lane == 0) {
        cnt[r] = c;
        if (r < n_pad) {
            const float h = (float)q;
            norm[r] = make_float2(h, (float)(q - (double)h));
            root[r] = __double2float_ru(sqrt(q));
        }
    }
}

__global__ void __launch_bounds__(256) k_sp_rows(const float *__restrict__ X, int64_t n, int32_t d,
                                                 const int32_t *__restrict__ rowptr, int64_t cap,
                                                 int32_t *__restrict__ rcol, float *__restrict__ rval, int32_t width,
                                                 float2 *__restrict__ ell) {
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (r >= n) return;
    int64_t base = rowptr[r];
    const int64_t first = base;
    float2 *sl = ell + (r >> 5) * width * 32 + (r & 31);
    for (int t0 = 0; t0 < d; t0 += 32) {
        const int t = t0 + lane;
        const float v = t < d ? X[r * d + t] : 0.0f;
        const unsigned m = __ballot_sync(0xffffffffu, v != 0.0f);
        const int64_t e = base + __popc(m & ((1u << lane) - 1u));
        if (v != 0.0f && e < cap) {
            rcol[e] = t;
            rval[e] = v;
            if (e - first < width) sl[(e - first) * 32] = make_float2(v, __int_as_float(t));
        }
        base += __popc(m);
    }
}

// one block per group of 32 rows: entries by dimension, then row
constexpr int SG_THREADS = 256;
__global__ void __launch_bounds__(SG_THREADS) k_sp_groups(int32_t d, const int32_t *__restrict__ rowptr,
                                                          const int32_t *__restrict__ rcol, const float *__restrict__ rval,
                                                          uint32_t *__restrict__ goff, float2 *__restrict__ gent) {
    extern __shared__ uint32_t off[];                    // [d]
    __shared__ uint32_t wsum[SG_THREADS / 32];
    const int64_t g = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int32_t e0 = rowptr[32 * g], e1 = rowptr[32 * g + 32];
    for (int t = tid; t < d; t += SG_THREADS) off[t] = 0u;
    __syncthreads();
    for (int32_t e = e0 + tid; e < e1; e += SG_THREADS) atomicAdd(off + rcol[e], 1u);
    __syncthreads();
    // exclusive sums, 256 dimensions at a time
    uint32_t carry = 0u;
    for (int t0 = 0; t0 < d; t0 += SG_THREADS) {
        const int t = t0 + tid;
        const uint32_t c = t < d ? off[t] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wp] = x;
        __syncthreads();
        uint32_t before = carry, total = 0u;
#pragma unroll
        for (int q = 0; q < SG_THREADS / 32; ++q) {
            if (q < wp) before += wsum[q];
            total += wsum[q];
        }
        if (t < d) {
            off[t] = before + x - c;
            goff[((g >> 2) * d + t) * 4 + (g & 3)] = (before + x - c) << 6 | c;
        }
        carry += total;
        __syncthreads();
    }
    for (int r = 0; r < 32; ++r) {
        const int32_t a = rowptr[32 * g + r], b = rowptr[32 * g + r + 1];
        for (int32_t e = a + tid; e < b; e += SG_THREADS) gent[e0 + off[rcol[e]]++] = make_float2(rval[e], __int_as_float(r));
        __syncthreads();
    }
}

constexpr int SD_LD = 65;                  // (an odd stride: the transposed read meets every bank)
__global__ void __launch_bounds__(256) k_sp_dist(SparseRows R, float *__restrict__ D, int64_t ld) {
    const int64_t I = blockIdx.y, J = blockIdx.x;
    if (J < 2 * I) return;
    __shared__ float S[128 * SD_LD];
    const int tid = threadIdx.x, c = tid & 63, q = tid >> 6;
    const int64_t row0 = I * 128, col0 = J * 64, j = col0 + c, g = 4 * I + q;
    float *own = S + (32 * q) * SD_LD + c;
    for (int r = 0; r < 32; ++r) own[r * SD_LD] = 0.0f;
    sparse_products(R, j, g, [&](float v, float2 x) {
        float *a = own + __float_as_int(x.y) * SD_LD;
        *a = fmaf(v, x.x, *a);
    });
    // (the average row's entries for all pairs, so that the two blocks of the
    // diagonal that write a pair's entry agree)
    const float nj = R.norm[j].x, cj = 0.03f / (5.9604645e-08f * (float)(R.width / 2 + 2));
    uint32_t canc = 0u;
    for (int r = 0; r < 32; ++r) {
        const int64_t i = row0 + 32 * q + r;
        const float nn = __fadd_rn(R.norm[i].x, nj);
        const float v = fmaxf(0.0f, fmaf(-2.0f, own[r * SD_LD], nn));
        own[r * SD_LD] = v;
        if (v * cj < nn) canc |= 1u << r;
        if (i < R.n && j < R.n) D[i * ld + j] = v;
    }
    // Rows close together and far from the origin (a dimension all rows hold,
    // with values far above the others'): their Gram form cancels, so the
    // distance comes from the lists' differences.  (From the Gram alone, 20,000 x
    // 2,048 with a column of 1,000s had every pair for a candidate: 964 ms a tree,
    // 22 so.)
    while (canc) {
        const int r = __ffs(canc) - 1;
        const int64_t i = row0 + 32 * q + r;
        canc &= canc - 1u;
        if (i == j || i >= R.n || j >= R.n) continue;
        float h, l;
        sparse_dist2(R, i, j, h, l);
        own[r * SD_LD] = D[i * ld + j] = __int_as_float(__float_as_int(h) | (int)0x80000000);
    }
    __syncthreads();
    for (int e = tid; e < 128 * 64; e += 256) {
        const int r = e & 127, cc = e >> 7;
        if (row0 + r < R.n && col0 + cc < R.n) D[(col0 + cc) * ld + row0 + r] = S[r * SD_LD + cc];
    }
}
}  // namespace

void SparseRows::carve(Arena &A, int64_t n_, int32_t d_, int64_t nnz) {
    n = n_;
    d = d_;
    n_pad = ceil_div(n, 128) * 128;
    cap = nnz;
    rowptr = A.take<int32_t>(n_pad + 1);
    cnt = A.take<int32_t>(n_pad + 1);
    tmp = A.take<int32_t>(scan_tmp_elems(n_pad + 1));
    rcol = A.take<int32_t>(nnz);
    rval = A.take<float>(nnz);
    goff = A.take<uint32_t>((size_t)(n_pad / 32) * d);
    gent = A.take<float2>(nnz);
    norm = A.take<float2>(n_pad);
    root = A.take<float>(n_pad);
    // rows up to twice the average length and a little wholly in slots
    width = (int32_t)(2 * ceil_div(nnz, n) + 8);
    ell = A.take<float2>((size_t)n_pad * width);
}

cudaError_t sparse_stats(const float *X, int64_t n, int32_t d, uint32_t *stat, cudaStream_t s) {
    const int64_t blocks = ceil_div(n, 8), cap = (int64_t)num_sms() * 8;
    k_sp_stats<<<(unsigned)(blocks < cap ? blocks : cap), 256, 0, ISO_S(s)>>>(X, n, d, stat);
    return cudaGetLastError();
}

// The dense kernels' work grows with d, these with the non-zeros (some 15
// instructions per look-up and product): from 1 in 16 on they win also where
// all rows hold the same dimensions.
bool sparse_pays(int64_t n, int32_t d, int64_t nnz, float norm_max) {
    return n >= 2 && d >= SPARSE_MIN_D && d <= SPARSE_MAX_D && nnz > 0 && nnz < (int64_t(1) << 31) && nnz <= n * d / 16 &&
           norm_max < 0x1p100f;
}

cudaError_t sparse_build(SparseRows &R, const float *X, cudaStream_t s) {
    cudaError_t e;
    k_sp_count<<<(unsigned)ceil_div(R.n_pad + 1, 8), 256, 0, ISO_S(s)>>>(X, R.n, R.n_pad, R.d, R.cnt, R.norm, R.root);
    if ((e = exclusive_scan_i32(R.cnt, R.rowptr, R.n_pad + 1, R.tmp, s))) return e;
    k_sp_rows<<<(unsigned)ceil_div(R.n, 8), 256, 0, ISO_S(s)>>>(X, R.n, R.d, R.rowptr, R.cap, R.rcol, R.rval, R.width, R.ell);
    static std::atomic<unsigned long long> seen{0};
    if (first_on_device(seen)) {
        if ((e = cudaFuncSetAttribute(k_sp_groups, cudaFuncAttributeMaxDynamicSharedMemorySize, SPARSE_MAX_D * 4))) return e;
        done_on_device(seen);
    }
    k_sp_groups<<<(unsigned)(R.n_pad / 32), SG_THREADS, (size_t)R.d * 4, ISO_S(s)>>>(R.d, R.rowptr, R.rcol, R.rval, R.goff,
                                                                                  R.gent);
    return cudaGetLastError();
}

cudaError_t sparse_dist(const SparseRows &R, float *D, int64_t ld, cudaStream_t s) {
    const dim3 g((unsigned)(R.n_pad / 64), (unsigned)(R.n_pad / 128));
    k_sp_dist<<<g, 256, 0, ISO_S(s)>>>(R, D, ld);
    return cudaGetLastError();
}

}  // namespace iso
