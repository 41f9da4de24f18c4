// weights64.cu -- eq. omega and eq. potential for FP64 input (and for FP32
// input with the FP64 option), in FP64 throughout.
//
// GB300's FP64 pipe issues 2 operations per clock per SM, 64 times fewer than
// FP32, and every pair needs 3 d + about 30 of them (subtract, multiply and
// add per dimension, separately rounded as in the canonical key, so that the
// exponent d / sigma carries the same roundings as the distances of the tree;
// root, quotient, exponential, sums): the pipe is the bound, so the kernel
// does each unordered pair once for both of its rows, over all SMs.  The
// first form (one thread per row, every column in turn) did each pair twice
// and filled n / 256 SMs only: at 2,000 x 8 its 8 blocks kept 144 SMs idle.
// Measured (omega stage): 20,011 x 24, 2 x 10^8 pairs, 38.1 ms (about 120
// operations per pair at the pipe's 629 G/s) against 155.5 ms before; 2,000 x
// 8: 0.25 ms against 8.4; 178 x 13: 0.024 against 0.72.
//
// Upper-triangle pairs (I, J) of TB-row tiles are the work items; row
// partials (rows of I) and column partials (rows of J) go to fixed slots of
// the item and are added in a fixed order, so the result is deterministic.
// TB = 16 up to 1,024 points (178 points: 78 items instead of 21, on as many
// SMs), else 32 (fewer partial sums: 100 MB at 20,011 points).
#include <math.h>

#include "common.cuh"

namespace iso {
namespace {
constexpr int W6_THREADS = 128;
constexpr int W6_DC = 32;                    // dimensions per shared-memory chunk
constexpr int W6_SMALL_N = 1024;             // tiles of 16 rows up to here
constexpr int W6_TAB = 512;

// ---- 2^(-j/512) as double-doubles, built at compile time: the Taylor series
// of exp in double-double arithmetic (Dekker's product, Knuth's sum).
struct DD {
    double h, l;
};
constexpr DD dd_fast(double a, double b) {
    const double s = a + b;
    return DD{s, b - (s - a)};
}
constexpr DD dd_sum(double a, double b) {
    const double s = a + b, t = s - a;
    return DD{s, (a - (s - t)) + (b - t)};
}
constexpr DD dd_prod(double a, double b) {
    const double p = a * b;
    const double ca = 134217729.0 * a, ah = ca - (ca - a), al = a - ah;
    const double cb = 134217729.0 * b, bh = cb - (cb - b), bl = b - bh;
    return DD{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD dd_add(DD a, DD b) {
    const DD s = dd_sum(a.h, b.h);
    return dd_fast(s.h, s.l + (a.l + b.l));
}
constexpr DD dd_mul(DD a, DD b) {
    const DD p = dd_prod(a.h, b.h);
    return dd_fast(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_div(DD a, double b) {
    const double q = a.h / b;
    const DD p = dd_prod(q, b);
    return dd_fast(q, ((a.h - p.h) - p.l + a.l) / b);
}
constexpr double LN2_H = 0x1.62e42fefa39efp-1, LN2_L = 0x1.abc9e3b39803fp-56;     // ln 2 to 107 bits
struct Exp64Table {
    double2 t[W6_TAB];
};
constexpr Exp64Table make_exp64() {
    Exp64Table T{};
    for (int j = 0; j < W6_TAB; ++j) {
        const DD x = dd_mul(DD{LN2_H, LN2_L}, DD{-(double)j / W6_TAB, 0.0});
        DD sum{1.0, 0.0}, term{1.0, 0.0};
        for (int k = 1; k <= 26; ++k) {
            term = dd_div(dd_mul(term, x), (double)k);
            sum = dd_add(sum, term);
        }
        T.t[j].x = sum.h;
        T.t[j].y = sum.l;
    }
    return T;
}
__device__ const Exp64Table g_exp64 = make_exp64();

// exp(-y), y >= 0: y = k ln2/512 + r with |r| <= ln2/1024 (table-driven
// reduction after Tang 1989; ln2/512 = C1 + C2, C1 with 33 significant bits,
// so k C1 is exact for k < 2^20), exp(-r) - 1 to degree 4 (the next term is
// below 1.2e-18), the table entry as a double-double.  10 FP64 operations.
// Past 700 the library's exp takes over (subnormal results).
constexpr double E6_C1 = 0x1.62e42fefp-10;
constexpr double E6_C2 = (LN2_H / W6_TAB - E6_C1) + LN2_L / W6_TAB;
__device__ __forceinline__ double exp_neg64(double y, const double2 *__restrict__ tab) {
    if (__double2hiint(y) >= 0x4085e000) return exp(-y);            // y >= 700, infinity, NaN
    const double magic = 6755399441055744.0;                       // 1.5 x 2^52
    const double tk = __fma_rn(y, (double)W6_TAB / LN2_H, magic);
    const int k = __double2loint(tk);
    const double kd = __dsub_rn(tk, magic);
    double r = __fma_rn(kd, -E6_C1, y);
    r = __fma_rn(kd, -E6_C2, r);
    double q = __fma_rn(r, 1.0 / 24.0, -1.0 / 6.0);
    q = __fma_rn(q, r, 0.5);
    q = __fma_rn(q, r, -1.0);
    q = __dmul_rn(q, r);
    const double2 t = tab[k & (W6_TAB - 1)];
    const double v = __dadd_rn(t.x, __fma_rn(t.x, q, t.y));
    return __hiloint2double(__double2hiint(v) - ((k / W6_TAB) << 20), __double2loint(v));
}

// Unordered tile pair w = (I, J), I <= J, of the upper triangle, row-major.
__device__ __forceinline__ void tri_pair(int64_t w, int64_t T, int64_t &I, int64_t &J) {
    const double b = 2.0 * (double)T + 1.0;
    int64_t i = (int64_t)floor((b - sqrt(b * b - 8.0 * (double)w)) * 0.5);
    if (i < 0) i = 0;
    while (i > 0 && i * T - i * (i - 1) / 2 > w) --i;
    while ((i + 1) * T - (i + 1) * i / 2 <= w) ++i;
    I = i;
    J = i + (w - (i * T - i * (i - 1) / 2));
}

// fast: sigma is far enough from the ends of the exponent range that the
// quotient dist / sigma may come from the reciprocal with two FMA corrections
// (Markstein's scheme: the second leaves the correctly rounded quotient).
template <class T, int TB, bool WITH_P>
__global__ void __launch_bounds__(W6_THREADS)
k_weights64(const T *__restrict__ X, int64_t n, int32_t d, int64_t ntiles, int64_t nitems, double sigma, double inv,
            int fast, double *__restrict__ part) {
    constexpr int RI = TB / 16, CJ = TB / 8;                        // a thread's rows and columns
    __shared__ double As[W6_DC][TB + 1], Bs[W6_DC][TB + 1];
    __shared__ double2 tab[W6_TAB];
    __shared__ double sc[WITH_P ? 2 : 1][4][TB];
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, lane = tid & 31, wp = tid >> 5;
    for (int q = tid; q < W6_TAB; q += W6_THREADS) tab[q] = g_exp64.t[q];
    for (int64_t w = blockIdx.x; w < nitems; w += gridDim.x) {
        int64_t I, J;
        tri_pair(w, ntiles, I, J);
        const int64_t row0 = I * TB, col0 = J * TB;
        double acc[RI][CJ];
#pragma unroll
        for (int i = 0; i < RI; ++i)
#pragma unroll
            for (int j = 0; j < CJ; ++j) acc[i][j] = 0.0;
        for (int32_t t0 = 0; t0 < d; t0 += W6_DC) {
            const int tl = d - t0 < W6_DC ? d - t0 : W6_DC;
            __syncthreads();
            for (int e = tid; e < TB * tl; e += W6_THREADS) {
                const int r = e / tl, t = e - r * tl;
                As[t][r] = row0 + r < n ? (double)X[(row0 + r) * d + t0 + t] : 0.0;
                Bs[t][r] = col0 + r < n ? (double)X[(col0 + r) * d + t0 + t] : 0.0;
            }
            __syncthreads();
#pragma unroll 2
            for (int t = 0; t < tl; ++t) {
                double a[RI], b[CJ];
#pragma unroll
                for (int i = 0; i < RI; ++i) a[i] = As[t][ty + 16 * i];
#pragma unroll
                for (int j = 0; j < CJ; ++j) b[j] = Bs[t][tx + 8 * j];
#pragma unroll
                for (int i = 0; i < RI; ++i)
#pragma unroll
                    for (int j = 0; j < CJ; ++j) {
                        const double df = __dsub_rn(a[i], b[j]);
                        acc[i][j] = __dadd_rn(acc[i][j], __dmul_rn(df, df));      // the canonical key's roundings
                    }
            }
        }
        double rw[RI], rp[RI], cw[CJ], cp[CJ];
#pragma unroll
        for (int i = 0; i < RI; ++i) { rw[i] = 0.0; rp[i] = 0.0; }
#pragma unroll
        for (int j = 0; j < CJ; ++j) { cw[j] = 0.0; cp[j] = 0.0; }
#pragma unroll
        for (int i = 0; i < RI; ++i) {
            const int64_t gr = row0 + ty + 16 * i;
#pragma unroll
            for (int j = 0; j < CJ; ++j) {
                const int64_t gc = col0 + tx + 8 * j;
                if (gr >= n || gc >= n || gr == gc) continue;
                const double dist = __dsqrt_rn(acc[i][j]);
                double y;
                if (fast && __double2hiint(dist) < 0x7ff00000) {
                    y = __dmul_rn(dist, inv);
                    y = __fma_rn(__fma_rn(-y, sigma, dist), inv, y);
                    y = __fma_rn(__fma_rn(-y, sigma, dist), inv, y);
                } else {
                    y = __ddiv_rn(dist, sigma);
                }
                const double f = exp_neg64(y, tab);
                rw[i] = __dadd_rn(rw[i], f);
                cw[j] = __dadd_rn(cw[j], f);
                if constexpr (WITH_P) {
                    rp[i] = __dadd_rn(rp[i], dist);
                    cp[j] = __dadd_rn(cp[j], dist);
                }
            }
        }
        // rows: over the 8 lanes of a row; columns: over the 4 row groups of
        // the warp, then the 4 warps (fixed trees)
        double *pr = part + w * (int64_t)((WITH_P ? 4 : 2) * TB);
#pragma unroll
        for (int i = 0; i < RI; ++i) {
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                rw[i] = __dadd_rn(rw[i], __shfl_xor_sync(0xffffffffu, rw[i], o));
                if constexpr (WITH_P) rp[i] = __dadd_rn(rp[i], __shfl_xor_sync(0xffffffffu, rp[i], o));
            }
            if (tx == 0) {
                pr[ty + 16 * i] = rw[i];
                if constexpr (WITH_P) pr[2 * TB + ty + 16 * i] = rp[i];
            }
        }
        if (I == J) continue;                                       // (the diagonal holds both orders of its pairs)
#pragma unroll
        for (int j = 0; j < CJ; ++j) {
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) {
                cw[j] = __dadd_rn(cw[j], __shfl_xor_sync(0xffffffffu, cw[j], o));
                if constexpr (WITH_P) cp[j] = __dadd_rn(cp[j], __shfl_xor_sync(0xffffffffu, cp[j], o));
            }
            if (lane < 8) {
                sc[0][wp][tx + 8 * j] = cw[j];
                if constexpr (WITH_P) sc[WITH_P ? 1 : 0][wp][tx + 8 * j] = cp[j];
            }
        }
        __syncthreads();
        for (int c = tid; c < (WITH_P ? 2 : 1) * TB; c += W6_THREADS) {
            const int k = c / TB, q = c - k * TB;
            pr[(2 * k + 1) * TB + q] = __dadd_rn(__dadd_rn(sc[k][0][q], sc[k][1][q]), __dadd_rn(sc[k][2][q], sc[k][3][q]));
        }
        __syncthreads();
    }
}

// Rows of tile I: the items (J, I), J < I (column partials) and (I, J), J >= I
// (row partials); 256 / TB groups of threads take every 256/TB-th J, their
// sums are added in group order.
template <int TB, bool WITH_P>
__global__ void __launch_bounds__(256) k_weights64_reduce(const double *__restrict__ part, int64_t n, int64_t ntiles,
                                                          double alpha, int include_self, double *__restrict__ omega,
                                                          double *__restrict__ pout) {
    constexpr int NG = 256 / TB, ST = (WITH_P ? 4 : 2) * TB;
    __shared__ double sw[NG][TB], sp[WITH_P ? NG : 1][TB];
    const int64_t I = blockIdx.x;
    const int c = threadIdx.x % TB, g = threadIdx.x / TB;
    double w = 0.0, p = 0.0;
#pragma unroll 4
    for (int64_t J = g; J < ntiles; J += NG) {
        const int64_t it = J < I ? J * ntiles - J * (J - 1) / 2 + (I - J) : I * ntiles - I * (I - 1) / 2 + (J - I);
        const double *pr = part + it * ST + (J < I ? TB : 0) + c;
        w = __dadd_rn(w, pr[0]);
        if constexpr (WITH_P) p = __dadd_rn(p, pr[2 * TB]);
    }
    sw[g][c] = w;
    if constexpr (WITH_P) sp[g][c] = p;
    __syncthreads();
    if (g != 0) return;
    const int64_t r = I * TB + c;
    if (r >= n) return;
    for (int q = 1; q < NG; ++q) {
        w = __dadd_rn(w, sw[q][c]);
        if constexpr (WITH_P) p = __dadd_rn(p, sp[q][c]);
    }
    omega[r] = include_self ? __dadd_rn(w, 1.0) : w;
    if (WITH_P && pout) pout[r] = __dmul_rn(alpha, p);
}

template <class T, int TB, bool WITH_P>
void launch64(const void *X, int64_t n, int32_t d, double sigma, double alpha, int include_self, double *omega,
              double *p, double *part, cudaStream_t s) {
    const int64_t T0 = ceil_div(n, TB), items = T0 * (T0 + 1) / 2, cap = (int64_t)num_sms() * 8;
    const double inv = 1.0 / sigma;
    const int fast = sigma > 0x1p-400 && sigma < 0x1p400;
    k_weights64<T, TB, WITH_P><<<(unsigned)(items < cap ? items : cap), W6_THREADS, 0, ISO_S(s)>>>(
        (const T *)X, n, d, T0, items, sigma, inv, fast, part);
    k_weights64_reduce<TB, WITH_P><<<(unsigned)T0, 256, 0, ISO_S(s)>>>(part, n, T0, alpha, include_self, omega, p);
}
}  // namespace

// Bytes of the items' partial sums.
size_t weights64_bytes(int64_t n, bool with_p) {
    const int64_t tb = n <= W6_SMALL_N ? 16 : 32, t = ceil_div(n, tb);
    return (size_t)(t * (t + 1) / 2) * (size_t)((with_p ? 4 : 2) * tb) * sizeof(double);
}

// part: weights64_bytes(n, alpha != 0 && p) bytes.
cudaError_t weights64_launch(const void *X, int64_t n, int32_t d, int dtype, double sigma, double alpha,
                             int include_self, double *omega, double *p, void *part, cudaStream_t s) {
    const bool wp = alpha != 0.0 && p, f64 = dtype == ISOCLUST_F64;
    double *q = (double *)part;
#define ISO_W64(TV, TBV)                                                                                \
    (wp ? launch64<TV, TBV, true>(X, n, d, sigma, alpha, include_self, omega, p, q, s)                  \
        : launch64<TV, TBV, false>(X, n, d, sigma, alpha, include_self, omega, p, q, s))
    if (n <= W6_SMALL_N) {
        if (f64) ISO_W64(double, 16); else ISO_W64(float, 16);
    } else {
        if (f64) ISO_W64(double, 32); else ISO_W64(float, 32);
    }
#undef ISO_W64
    if (!wp && p) {
        cudaError_t e = cudaMemsetAsync(p, 0, sizeof(double) * n, s);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}
}  // namespace iso
