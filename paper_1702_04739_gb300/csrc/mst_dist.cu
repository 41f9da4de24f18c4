// mst_dist.cu -- Boruvka rounds on stored distances.
//
// Section 3.5's minimum spanning tree for sets whose FP32 distance matrix is
// worth keeping: every round then reads the matrix instead of forming n^2
// products again, and needs neither the sweep's row data (mean, order, BF16
// split, norms, maps) nor its candidate lists.  A round of short rows is two
// launches: k_dist_scan (a block per row: minimum over the other components'
// columns, then every column within the error margin keyed in FP64, the
// row's best into its component's minimum) and k_union (one block: pairs,
// hooks, pointers, labels, edges).  Bound by the matrix: n^2 words written
// once and read once a round (from L2 for up to about 5,000 points), then by
// the two launches and the host's question whether the forest is complete.
#include <math.h>

#include "mst.cuh"
#include "sparse.cuh"

namespace iso {
namespace {
constexpr int TPB = 256;

__device__ __forceinline__ bool dist_active(const int32_t *c) { return c[MC_NCOMP] > c[MC_TARGET]; }

// FP32 squared distances of one pair of 64-row tiles, 4 x 4 pairs per thread,
// both halves of the matrix written.  Differences are rounded once (FP64
// points: differences of the points times sc, a power of two, so that FP32
// holds their squares), squares and sums are FMAs: relative error at most
// (d + 3) 2^-24 and an underflow term.
constexpr int DS_T = 64, DS_K = 32;
template <class P>
__global__ void __launch_bounds__(256) k_dist_tiles(const P *__restrict__ X, int64_t n, int32_t d, double sc, int64_t T,
                                                    float *__restrict__ D, int64_t ld) {
    __shared__ __align__(16) P As[DS_K][DS_T + 16 / sizeof(P)];
    __shared__ __align__(16) P Bs[DS_K][DS_T + 16 / sizeof(P)];
    // item -> (I, J), I <= J
    const int64_t w = blockIdx.x;
    const double q = 2.0 * (double)T + 1.0;
    int64_t I = (int64_t)floor((q - sqrt(q * q - 8.0 * (double)w)) * 0.5);
    if (I < 0) I = 0;
    while (I > 0 && I * T - I * (I - 1) / 2 > w) --I;
    while ((I + 1) * T - (I + 1) * I / 2 <= w) ++I;
    const int64_t J = I + (w - (I * T - I * (I - 1) / 2));
    const int64_t row0 = I * DS_T, col0 = J * DS_T;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
    for (int t0 = 0; t0 < d; t0 += DS_K) {
        const int tl = d - t0 < DS_K ? d - t0 : DS_K;
        __syncthreads();
        for (int e = tid; e < DS_T * DS_K; e += 256) {
            const int r = e / DS_K, t = e % DS_K;
            P a = P(0), b = P(0);
            if (t < tl) {
                if (row0 + r < n) a = X[(row0 + r) * d + t0 + t];
                if (col0 + r < n) b = X[(col0 + r) * d + t0 + t];
            }
            if constexpr (sizeof(P) == 8) {
                a *= sc;
                b *= sc;
            }
            As[t][r] = a;
            Bs[t][r] = b;
        }
        __syncthreads();
#pragma unroll 8
        for (int t = 0; t < tl; ++t) {
            __align__(16) P a[4], b[4];
            constexpr int V = 16 / sizeof(P);                // 16-byte loads
#pragma unroll
            for (int i = 0; i < 4; i += V) {
                *reinterpret_cast<float4 *>(a + i) = *reinterpret_cast<const float4 *>(&As[t][ty * 4 + i]);
                *reinterpret_cast<float4 *>(b + i) = *reinterpret_cast<const float4 *>(&Bs[t][tx * 4 + i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float df = (float)(a[i] - b[j]);
                    acc[i][j] = __fmaf_rn(df, df, acc[i][j]);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4 *>(D + (row0 + ty * 4 + i) * ld + col0 + tx * 4) =
            make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (I == J) return;
    // the other half through shared memory, so that it leaves in whole lines
    static_assert(sizeof(As) >= DS_T * DS_K * sizeof(float), "half a transposed tile");
    float(*S)[DS_T] = reinterpret_cast<float(*)[DS_T]>(&As[0][0]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        __syncthreads();
        if ((tx >> 3) == h)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) S[(tx & 7) * 4 + j][ty * 4 + i] = acc[i][j];
        __syncthreads();
        for (int e = tid; e < 32 * 16; e += 256) {
            const int r = e >> 4, c = e & 15;
            *reinterpret_cast<float4 *>(D + (col0 + 32 * h + r) * ld + row0 + 4 * c) =
                *reinterpret_cast<const float4 *>(&S[r][4 * c]);
        }
    }
}

// One row per block.  INLINE (short rows): a thread keys its own columns, the
// block's best goes to rowd2 / rowj and to its component's minimum.  Else the
// columns go to surv for the FP64 keys of long rows, more than TC_SURV of them
// (exact ties) to the rescan.
constexpr int DSC_THREADS = 128;
template <class P, bool INLINE>
__global__ void __launch_bounds__(DSC_THREADS) k_dist_scan(const P *__restrict__ X, int64_t n, int32_t d,
                                                           const float *__restrict__ D, int64_t ld, float mul, float add,
                                                           const int32_t *__restrict__ comp, double *__restrict__ rowd2,
                                                           int32_t *__restrict__ rowj, unsigned long long *__restrict__ cd2,
                                                           int32_t *__restrict__ nsurv, int32_t *__restrict__ surv,
                                                           int32_t *__restrict__ ovf, int32_t *counters) {
    if (!dist_active(counters)) return;
    __shared__ float smin[DSC_THREADS / 32];
    __shared__ double sb[DSC_THREADS / 32];
    __shared__ int32_t sj[DSC_THREADS / 32];
    __shared__ int scnt;
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int64_t i = blockIdx.x;
    const int32_t ci = comp[i];
    const float *row = D + i * ld;
    const int64_t n4 = n & ~(int64_t)3;
    if (tid == 0) scnt = 0;
    float m = INFINITY;
    for (int64_t j = 4 * tid; j < n4; j += 4 * DSC_THREADS) {
        const float4 v = *reinterpret_cast<const float4 *>(row + j);
        const int4 c = *reinterpret_cast<const int4 *>(comp + j);
        if (c.x != ci) m = fminf(m, v.x);
        if (c.y != ci) m = fminf(m, v.y);
        if (c.z != ci) m = fminf(m, v.z);
        if (c.w != ci) m = fminf(m, v.w);
    }
    if (n4 + tid < n && comp[n4 + tid] != ci) m = fminf(m, row[n4 + tid]);
    const float low = m;                   // (a thread whose own columns hold none does not look again)
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smin[wp] = m;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < DSC_THREADS / 32; ++q) m = fminf(m, smin[q]);
    const float thr = __fadd_ru(__fmul_ru(m, mul), add);
    double best = INFINITY;
    int32_t bestj = -1;
    auto see = [&](int64_t j) {
        if constexpr (INLINE) {
            double e = 0.0;
            for (int t = 0; t < d; ++t) {
                const double df = __dsub_rn((double)X[i * d + t], (double)X[j * d + t]);
                e = __dadd_rn(e, __dmul_rn(df, df));
            }
            if (bestj < 0 || key_less(e, (int32_t)i, (int32_t)j, best, (int32_t)i, bestj)) {
                best = e;
                bestj = (int32_t)j;
            }
        } else {
            const int q = atomicAdd(&scnt, 1);
            if (q < TC_SURV) surv[i * TC_SURV + q] = (int32_t)j;
        }
    };
    if (low <= thr)
        for (int64_t j = 4 * tid; j < n4; j += 4 * DSC_THREADS) {
            const float4 v = *reinterpret_cast<const float4 *>(row + j);
            if (fminf(fminf(v.x, v.y), fminf(v.z, v.w)) > thr) continue;
            const int4 c = *reinterpret_cast<const int4 *>(comp + j);
            if (c.x != ci && v.x <= thr) see(j);
            if (c.y != ci && v.y <= thr) see(j + 1);
            if (c.z != ci && v.z <= thr) see(j + 2);
            if (c.w != ci && v.w <= thr) see(j + 3);
        }
    if (n4 + tid < n && comp[n4 + tid] != ci && row[n4 + tid] <= thr) see(n4 + tid);
    if constexpr (INLINE) {
        auto take = [&](double e, int32_t j) {
            if (j >= 0 && (bestj < 0 || key_less(e, (int32_t)i, j, best, (int32_t)i, bestj))) {
                best = e;
                bestj = j;
            }
        };
        for (int o = 16; o > 0; o >>= 1) {
            const double e = __shfl_xor_sync(0xffffffffu, best, o);
            const int32_t j = __shfl_xor_sync(0xffffffffu, bestj, o);
            take(e, j);
        }
        if (lane == 0) {
            sb[wp] = best;
            sj[wp] = bestj;
        }
        __syncthreads();
        if (tid == 0) {
            for (int q = 1; q < DSC_THREADS / 32; ++q) take(sb[q], sj[q]);
            rowd2[i] = best;
            rowj[i] = bestj;
            if (bestj >= 0) atomicMin(cd2 + ci, dbits(best));
        }
    } else {
        __syncthreads();
        if (tid == 0) {
            nsurv[i] = scnt;
            rowj[i] = -1;
            if (scnt > TC_SURV) {
                ovf[atomicAdd(counters + MC_OVERFLOW, 1)] = (int32_t)i;
                rowj[i] = -2;
            }
        }
    }
}

// The scan for rows as lists: the distances come from a Gram, so a column is a
// candidate when the smallest distance its entry stands for is at most the
// smallest of the row's largest.  A product of rows takes a rounding per
// dimension both hold, at most k = the entries of row i, of a partial sum below
// |x_i| |x_j|, twice; the norms and the three last operations take one each of
// |x_i|^2 + |x_j|^2 (v is at most twice that): within 2^-24 (2 k |x_i| |x_j| + 4
// (|x_i|^2 + |x_j|^2)), and 10 % above; an entry with its sign set is a direct
// sum, within one rounding of itself.  (With the longest row's entries for
// every pair and half the norms for the product, one full row of ones among
// 50,000 of 41 entries had every column for a candidate: 29 ms -> 990.)
// Keys from the lists (a dimension that neither row holds adds nothing to the
// key), by a warp per candidate: the lanes find each entry's place in the two
// lists' common order and leave its square there, one adds them up.  (One
// thread walking the lists, in global or in shared memory: some 10 us of
// latency a key, 6 ms a round at 50,000 x 4,096.)  Only a thread whose own
// columns hold two candidates or more looks at them again.
constexpr int SC_THREADS = 512, SC_CAND = 128, SC_LIST = 128;
__global__ void __launch_bounds__(SC_THREADS) k_sparse_scan(const SparseRows R, int64_t n, const float *__restrict__ D,
                                                            int64_t ld, float add,
                                                            const int32_t *__restrict__ comp, double *__restrict__ rowd2,
                                                            int32_t *__restrict__ rowj,
                                                            unsigned long long *__restrict__ cd2, int32_t *counters) {
    if (!dist_active(counters)) return;
    constexpr int NW = SC_THREADS / 32;
    __shared__ float smin[NW];
    __shared__ double sb[NW];
    __shared__ int32_t sj[NW], scand[SC_CAND];
    __shared__ int scnt;
    __shared__ int32_t ac[SC_LIST], bc[NW][SC_LIST];
    __shared__ float av[SC_LIST], bv[NW][SC_LIST];
    __shared__ double sq[NW][2 * SC_LIST];
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int64_t i = blockIdx.x;
    const int32_t ci = comp[i];
    const float *row = D + i * ld;
    const float ri = R.root[i];
    const int32_t a0 = R.rowptr[i], alen = R.rowptr[i + 1] - a0;
    constexpr float U = 1.1f * 5.9604645e-08f;
    const float gk = __fmul_ru(__fmul_ru(2.0f * U, (float)(alen + 1)), ri), gn = 5.0f * U, own = __fmul_ru(gn, __fmul_ru(ri, ri));
    for (int e = tid; e < alen && e < SC_LIST; e += SC_THREADS) {
        ac[e] = R.rcol[a0 + e];
        av[e] = R.rval[a0 + e];
    }
    if (tid == 0) scnt = 0;
    const int64_t n4 = n & ~(int64_t)3;
    auto wide = [&](float rj) { return __fmaf_ru(rj, __fmaf_ru(gn, rj, gk), own); };
    // the thread's two smallest, and the column of the smaller
    float m = INFINITY, low = INFINITY, low2 = INFINITY;
    int32_t lowj = -1;
    auto margin = [&](float v, float rj) { return __float_as_int(v) < 0 ? __fmul_ru(-2.0f * U, v) : wide(rj); };
    auto first = [&](float v, float w, int64_t j) {
        const float l = __fsub_rd(v, w);
        m = fminf(m, __fadd_ru(v, w));
        low2 = fminf(low2, fmaxf(low, l));
        if (l < low) {
            low = l;
            lowj = (int32_t)j;
        }
    };
#pragma unroll 4
    for (int64_t j = 4 * tid; j < n4; j += 4 * SC_THREADS) {
        const float4 v = *reinterpret_cast<const float4 *>(row + j);
        const int4 c = *reinterpret_cast<const int4 *>(comp + j);
        const float4 q = *reinterpret_cast<const float4 *>(R.root + j);
        if ((__float_as_int(v.x) | __float_as_int(v.y) | __float_as_int(v.z) | __float_as_int(v.w)) >= 0) {
            if (c.x != ci) first(v.x, wide(q.x), j);
            if (c.y != ci) first(v.y, wide(q.y), j + 1);
            if (c.z != ci) first(v.z, wide(q.z), j + 2);
            if (c.w != ci) first(v.w, wide(q.w), j + 3);
        } else {                               // (a direct sum among them)
            if (c.x != ci) first(fabsf(v.x), margin(v.x, q.x), j);
            if (c.y != ci) first(fabsf(v.y), margin(v.y, q.y), j + 1);
            if (c.z != ci) first(fabsf(v.z), margin(v.z, q.z), j + 2);
            if (c.w != ci) first(fabsf(v.w), margin(v.w, q.w), j + 3);
        }
    }
    if (n4 + tid < n && comp[n4 + tid] != ci)
        first(fabsf(row[n4 + tid]), margin(row[n4 + tid], R.root[n4 + tid]), n4 + tid);
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smin[wp] = m;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NW; ++q) m = fminf(m, smin[q]);
    const float thr = __fadd_ru(m, add);
    double best = INFINITY;
    int32_t bestj = -1;
    auto take = [&](double e, int32_t j) {
        if (j >= 0 && (bestj < 0 || key_less(e, (int32_t)i, j, best, (int32_t)i, bestj))) {
            best = e;
            bestj = j;
        }
    };
    // the key along two lists, smallest dimension first
    auto key = [&](const int32_t *xc, const float *xv, int xn, const int32_t *yc, const float *yv, int yn) {
        double e = 0.0;
        int a = 0, b = 0;
        int32_t ta = xn > 0 ? xc[0] : INT32_MAX, tb = yn > 0 ? yc[0] : INT32_MAX;
        while (a < xn || b < yn) {
            double df = 0.0;
            const bool ua = ta <= tb, ub = tb <= ta;
            if (ua) {
                df = (double)xv[a++];
                ta = a < xn ? xc[a] : INT32_MAX;
            }
            if (ub) {
                df = __dsub_rn(df, (double)yv[b++]);
                tb = b < yn ? yc[b] : INT32_MAX;
            }
            e = __dadd_rn(e, __dmul_rn(df, df));
        }
        return e;
    };
    auto see = [&](int64_t j) {
        const int q = atomicAdd(&scnt, 1);
        if (q < SC_CAND) {
            scand[q] = (int32_t)j;
        } else {                                         // (many ties: by the thread itself)
            const int32_t b0 = R.rowptr[j];
            take(key(R.rcol + a0, R.rval + a0, alen, R.rcol + b0, R.rval + b0, R.rowptr[j + 1] - b0), (int32_t)j);
        }
    };
    auto again = [&](float v, float rj, int32_t c, int64_t j) {
        if (c != ci && __fsub_rd(fabsf(v), margin(v, rj)) <= thr) see(j);
    };
    if (low <= thr && low2 > thr) {
        see(lowj);
    } else if (low <= thr) {
        for (int64_t j = 4 * tid; j < n4; j += 4 * SC_THREADS) {
            const float4 v = *reinterpret_cast<const float4 *>(row + j);
            const int4 c = *reinterpret_cast<const int4 *>(comp + j);
            const float4 q = *reinterpret_cast<const float4 *>(R.root + j);
            again(v.x, q.x, c.x, j);
            again(v.y, q.y, c.y, j + 1);
            again(v.z, q.z, c.z, j + 2);
            again(v.w, q.w, c.w, j + 3);
        }
        if (n4 + tid < n) again(row[n4 + tid], R.root[n4 + tid], comp[n4 + tid], n4 + tid);
    }
    __syncthreads();
    const int nc = scnt < SC_CAND ? scnt : SC_CAND;
    if (tid == 0 && scnt > SC_CAND) atomicAdd(counters + MC_OVERFLOW, 1);      // (the call's count of such rows)
    for (int q = wp; q < nc; q += NW) {
        const int32_t j = scand[q], b0 = R.rowptr[j], blen = R.rowptr[j + 1] - b0;
        const bool fits = alen <= SC_LIST && blen <= SC_LIST;
        __syncwarp();
        if (fits)
            for (int e = lane; e < blen; e += 32) {
                bc[wp][e] = R.rcol[b0 + e];
                bv[wp][e] = R.rval[b0 + e];
            }
        __syncwarp();
        if (fits) {
            // entries of a list below t (or up to it)
            auto below = [](const int32_t *l, int n_, int32_t t) {
                int lo = 0, hi = n_;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (l[mid] < t) lo = mid + 1; else hi = mid;
                }
                return lo;
            };
            for (int e = lane; e < alen; e += 32) {
                const int p = below(bc[wp], blen, ac[e]);
                const double df = p < blen && bc[wp][p] == ac[e] ? __dsub_rn((double)av[e], (double)bv[wp][p]) : (double)av[e];
                sq[wp][e + p] = __dmul_rn(df, df);
            }
            for (int e = lane; e < blen; e += 32) {
                const int p = below(ac, alen, bc[wp][e] + 1);       // a dimension of both: the other list's entry, then a zero
                const bool both = p > 0 && ac[p - 1] == bc[wp][e];
                const double df = (double)bv[wp][e];
                sq[wp][e + p] = both ? 0.0 : __dmul_rn(df, df);
            }
            __syncwarp();
            double e = 0.0;
            for (int k = 0; k < alen + blen; ++k) e = __dadd_rn(e, sq[wp][k]);
            if (lane == 0) take(e, j);
        } else if (lane == 0) {
            take(key(R.rcol + a0, R.rval + a0, alen, R.rcol + b0, R.rval + b0, blen), j);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double e = __shfl_xor_sync(0xffffffffu, best, o);
        const int32_t j = __shfl_xor_sync(0xffffffffu, bestj, o);
        take(e, j);
    }
    if (lane == 0) {
        sb[wp] = best;
        sj[wp] = bestj;
    }
    __syncthreads();
    if (tid == 0) {
        for (int q = 1; q < NW; ++q) take(sb[q], sj[q]);
        rowd2[i] = best;
        rowj[i] = bestj;
        if (bestj >= 0) atomicMin(cd2 + ci, dbits(best));
    }
}

__global__ void k_dist_init(int32_t *__restrict__ comp, unsigned long long *__restrict__ cd2,
                            unsigned long long *__restrict__ cpair, int32_t *__restrict__ perm, int64_t n,
                            int32_t *counters) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v < 8) counters[v] = v == MC_NCOMP ? (int32_t)n : (v == MC_TARGET ? 1 : 0);
    if (v >= n) return;
    comp[v] = (int32_t)v;
    cd2[v] = cpair[v] = ~0ull;
    if (perm) perm[v] = (int32_t)v;          // (rows of the long rows' keys are points)
}

// The union step of a round by one block: the same steps as the kernels of
// the larger rounds (component minima's pairs, hooks, pointers to the roots,
// labels), with block barriers between them instead of launches (8 of them,
// some 3 us each, where a step over 5,000 points takes 1 us).
constexpr int UN_THREADS = 1024;
__global__ void __launch_bounds__(UN_THREADS) k_union(int32_t *comp, const double *__restrict__ rowd2,
                                                      const int32_t *__restrict__ rowj, int32_t n,
                                                      unsigned long long *cd2, unsigned long long *cpair, int32_t *tgt,
                                                      int32_t *nxt, int32_t *__restrict__ eu, int32_t *__restrict__ ev,
                                                      double *__restrict__ ed2, int32_t *counters, uint32_t *st) {
    if (!dist_active(counters)) return;
    __shared__ int sroots, sedges;
    const int tid = threadIdx.x;
    if (tid == 0) {
        sroots = 0;
        sedges = counters[MC_NEDGES];
    }
    for (int i = tid; i < n; i += UN_THREADS) {
        const int32_t j = rowj[i];
        if (j < 0) continue;
        const int32_t c = comp[i];
        if (dbits(rowd2[i]) != cd2[c]) continue;
        const unsigned long long a = (unsigned long long)min(i, j), b = (unsigned long long)max(i, j);
        atomicMin(cpair + c, (a << 32) | b);
    }
    __threadfence_block();
    __syncthreads();
    for (int v = tid; v < n; v += UN_THREADS) {
        if (comp[v] != v) continue;
        const unsigned long long pr = __ldcg(cpair + v);
        int32_t t = v;
        if (pr != ~0ull) {
            const int32_t a = (int32_t)(pr >> 32), b = (int32_t)(pr & 0xffffffffu);
            t = comp[comp[a] == v ? b : a];
        }
        tgt[v] = t;
    }
    __syncthreads();
    for (int v = tid; v < n; v += UN_THREADS) {
        if (comp[v] != v) continue;
        const int32_t T = tgt[v];
        if (T == v) {
            nxt[v] = v;
            continue;
        }
        const bool mutual = tgt[T] == v;
        nxt[v] = mutual && v < T ? v : T;
        if (!mutual || v < T) {
            const int q = atomicAdd(&sedges, 1);
            if (q < n - 1) {
                const unsigned long long pr = __ldcg(cpair + v);
                eu[q] = (int32_t)(pr >> 32);
                ev[q] = (int32_t)(pr & 0xffffffffu);
                ed2[q] = bitsd(cd2[v]);
            } else {
                atomicOr(st, DEV_EDGE_COUNT);
            }
        }
    }
    __syncthreads();
    // roots: find with path halving (every entry holds an ancestor throughout)
    volatile int32_t *vn = nxt;
    for (int v = tid; v < n; v += UN_THREADS) {
        if (comp[v] != v) continue;
        int32_t x = v;
        for (int it = 0;; ++it) {
            const int32_t p = vn[x];
            const int32_t q = p >= 0 && p < n ? vn[p] : -1;
            if (q < 0 || q >= n || it > n) {
                atomicOr(st, DEV_INTERNAL);
                break;
            }
            if (q == p) {
                vn[v] = p;
                break;
            }
            atomicCAS(reinterpret_cast<int *>(nxt) + x, p, q);
            x = q;
        }
    }
    __syncthreads();
    int roots = 0;
    for (int v = tid; v < n; v += UN_THREADS) {
        const int32_t r = vn[comp[v]];
        comp[v] = r;
        roots += r == v;
        cd2[v] = cpair[v] = ~0ull;
    }
    for (int o = 16; o > 0; o >>= 1) roots += __shfl_xor_sync(0xffffffffu, roots, o);
    if ((tid & 31) == 0 && roots) atomicAdd(&sroots, roots);
    __syncthreads();
    if (tid == 0) {
        counters[MC_NEDGES] = sedges;
        counters[MC_NCOMP] = sroots;
        counters[MC_ROUNDS] += 1;
        counters[MC_OVF_TOTAL] += counters[MC_OVERFLOW];
        counters[MC_OVERFLOW] = 0;
    }
}
}  // namespace

size_t mst_dist_bytes(int64_t n) {
    const int64_t p = ceil_div(n, DS_T) * DS_T;
    return (size_t)p * (size_t)p * sizeof(float);
}

// The stage in ms, stored distances / tensor-core sweep (blobs):
//   n      d = 2      24         64         128        512        1,500
//   180    .17/.48    .16/.44    .22/.51    .25/.56    .49/1.0    .91/1.9
//   2,000  .27/.65    .33/.59    .30/.58    .37/.69    .84/2.0    2.2/6.9
//   4,900  .47/.83    .55/.79    .59/.88    .71/1.04   1.5/3.0    4.0/25
//   6,144  .60/.85    .69/.80    .74/.94    .93/1.16   2.1/3.7    6.0/36
// (8,192 x 64 is even, x 256 2.4/2.2 before the keys of long rows were made
// faster.)  FP64 differences run at a 64th of the FP32 rate: 2,000 x 24 .49/.62,
// 4,900 x 2 .58/.83, x 8 .85/.85.
constexpr int64_t MST_DIST_MAX_N = 6144;
constexpr int64_t MST_DIST_MAX_F64 = 100000000;        // n^2 d
// Keys by the scan itself up to here (64 dimensions: 180 points .19 ms, with
// kernels of their own .22; 4,900 .88, .59)
constexpr int32_t MST_DIST_INLINE_MAX_D = 32;

// Rows by their non-zeros: while the matrix stays within 16 GiB.
bool mst_dist_sparse_wanted(int64_t n) { return n <= 65536; }

bool mst_dist_wanted(int64_t n, int32_t d, int dtype) {
    if (n < 2 || n > MST_DIST_MAX_N) return false;
    return dtype == ISOCLUST_F32 || (d <= 2 * MST_DIST_INLINE_MAX_D && n * n <= MST_DIST_MAX_F64 / d);
}

cudaError_t mst_build_dist(MstScratch &S, TcScratch &T, float *D, const void *X, int64_t n, int32_t d, int dtype,
                           int scale_exp, uint32_t *status, cudaStream_t s, const SparseRows *sp) {
    const int64_t Tn = ceil_div(n, DS_T), ld = Tn * DS_T;
    const unsigned tiles = (unsigned)(Tn * (Tn + 1) / 2);
    const bool f64 = dtype == ISOCLUST_F64, inl = sp || f64 || d <= MST_DIST_INLINE_MAX_D;
    const double sc = f64 ? ldexp(1.0, -scale_exp) : 1.0;
    cudaError_t e;
    k_dist_init<<<(unsigned)ceil_div(n < 8 ? 8 : n, TPB), TPB, 0, ISO_S(s)>>>(S.comp, S.cd2, S.cpair, inl ? nullptr : T.permp, n,
                                                                            S.counters);
    if (sp) {
        if ((e = sparse_dist(*sp, D, ld, s))) return e;
    } else if (f64)
        k_dist_tiles<double><<<tiles, 256, 0, ISO_S(s)>>>((const double *)X, n, d, sc, Tn, D, ld);
    else
        k_dist_tiles<float><<<tiles, 256, 0, ISO_S(s)>>>((const float *)X, n, d, sc, Tn, D, ld);
    // any column within m (1 + e) / (1 - e) + 2 add of the row's FP32 minimum
    // can hold the exact best (e: 10 % above the bound of the distances)
    const double u = 5.9604644775390625e-08, er = 1.1 * (double)(d + 3) * u;
    const double mul = (1.0 + er) / (1.0 - er), add = (double)(d + 1) * 1.401298464324817e-45 * 4.0;
    const float mul32 = (float)(mul * (1.0 + 1e-6)), add32 = (float)(2.01 * add) + 1.401298464324817e-45f;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(s, &cs))) return e;
    const bool ask = cs == cudaStreamCaptureStatusNone;
    int R = 1;                                         // components at least halve per round
    while ((int64_t(1) << (R - 1)) < n) ++R;
    for (int r = 0; r < R; ++r) {
#define ISO_SCAN(PT, INL)                                                                                              \
    k_dist_scan<PT, INL><<<(unsigned)n, DSC_THREADS, 0, ISO_S(s)>>>((const PT *)X, n, d, D, ld, mul32, add32, S.comp,   \
                                                                    S.rowd2, S.rowj, S.cd2, T.nsurv, T.surv,           \
                                                                    S.ovf_rows, S.counters)
        if (sp) {
            k_sparse_scan<<<(unsigned)n, SC_THREADS, 0, ISO_S(s)>>>(*sp, n, D, ld, add32, S.comp, S.rowd2, S.rowj, S.cd2,
                                                                   S.counters);
        } else if (f64) {
            ISO_SCAN(double, true);
        } else if (inl) {
            ISO_SCAN(float, true);
        } else {
            ISO_SCAN(float, false);
            if ((e = tc_key_rows(T, S, (const float *)X, n, d, mul, add, s))) return e;
            if ((e = mst_component_minima(S, n, s))) return e;
        }
#undef ISO_SCAN
        k_union<<<1, UN_THREADS, 0, ISO_S(s)>>>(S.comp, S.rowd2, S.rowj, (int32_t)n, S.cd2, S.cpair, S.tgt, S.nxt, S.eu,
                                                S.ev, S.ed2, S.counters, status);
        // (the first rounds seldom complete the forest: a round more that
        // returns at once costs less than the question)
        if (ask && r >= 1 && r + 1 < R) {
            int32_t h[8];
            if ((e = cudaMemcpyAsync(h, S.counters, sizeof(h), cudaMemcpyDeviceToHost, s))) return e;
            if ((e = cudaStreamSynchronize(s))) return e;
            if (h[MC_NCOMP] <= h[MC_TARGET]) break;
        }
    }
    return cudaGetLastError();
}

}  // namespace iso
