// Rayleigh quotients x^T A x / x^T B x of a block of vectors over the CSR pattern of
// A union B, in double-double arithmetic: the eigenvalues a probe returns (after Alg. 2).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sss {

// ---------------------------------------------------------------- Rayleigh quotients
// Error-free transformations (Knuth's TwoSum, the FMA form of Dekker's TwoProduct) and the
// compensated dot product of Ogita, Rump and Oishi ("Accurate sum and dot product", SIAM
// J. Sci. Comput. 2005): the sum is accumulated as hi + lo, every rounding error of a
// product or an addition carried into lo.
struct DD {
    double hi, lo;
};
__device__ __forceinline__ void dd_add_prod(DD &s, double a, double b) {
    const double p = a * b, pe = fma(a, b, -p);
    const double t = s.hi + p, z = t - s.hi;
    const double se = (s.hi - (t - z)) + (p - z);
    s.hi = t;
    s.lo += se + pe;
}
__device__ __forceinline__ void dd_add(DD &s, double hi, double lo) {
    const double t = s.hi + hi, z = t - s.hi;
    const double se = (s.hi - (t - z)) + (hi - z);
    s.hi = t;
    s.lo += se + lo;
}

// The products run in integers: double-double arithmetic takes some 20 FP64 operations per stored
// entry and column at 2 a clock and SM, a 64 x 64-bit multiply-add into 128 bits some ten at 64.
// Column c of X becomes x~ = round(x 2^(xbits - E_c)), |x| < 2^E_c, xbits 53 (fewer for rows of more
// than 4,096 entries): the quotient of x~ differs from that of x by the residual times the rounding
// (second order, below 1e-20, near convergence), as long as numerator and denominator share x~.  A row of A (of B) becomes round(a 2^(61 - E_i)): relative to the row's
// largest entry, 2^-62, below double-double's use for the dot products that follow.  Sums over a row
// are exact: 2^(61 + xbits) times its entries stays below 2^127.  The column's scale cancels in the
// quotient.  "Largest" is meant after a scaling by powers of two that follows the basis: x_i is
// multiplied by 2^s_i and column i of A and B by 2^-s_i, s_i as for the solves (k_fold_scales), so a pencil
// S A S, S B S gives the bits of A, B.  Gaussian pencil of 720 rows scaled by 2^-15 .. 2^15, vectors
// before convergence, error of a quotient of 0.5: 1.5e-8 without s_i, 9.5e-17 with it.
// N = 5,280, k = 112: 15 ms with double-double products, 1.5 ms now.

constexpr int kRqZero = -(1 << 20), kRqNan = 1 << 20;   // "exponents" of zero and of a non-finite value

// biased exponent of v 2^sh
__device__ __forceinline__ int rq_exp(double v, int sh) {
    const int ex = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
    return ex == 0 ? kRqZero : ex == 0x7ff ? kRqNan : ex + sh;
}
// round(v 2^(sh + bits - E)) for |v| 2^sh < 2^E, E = em - 1022, em >= rq_exp(v, sh)
__device__ __forceinline__ long long rq_fixed(double v, int sh, int em, int bits) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((b >> 52) & 0x7ff) + sh;
    if ((b >> 52 & 0x7ff) == 0) return 0;
    // v 2^sh = m 2^(ex - 1075), so v 2^(bits - em + 1022) = m 2^9 2^-(em - ex + 62 - bits)
    unsigned long long m = ((b & ((1ull << 52) - 1)) | (1ull << 52)) << 9;
    const int rs = min(em - ex + 62 - bits, 63);
    m = ((m >> (rs - 1)) + 1) >> 1;                 // rs >= 1: bits <= 61
    return (long long)b < 0 ? -(long long)m : (long long)m;
}

// em[c] = largest biased exponent of column c, row i times 2^sc[i] (kRqZero or less on entry)
__global__ void k_rq_colmax(int64_t n, int k, const double *__restrict__ X, const int32_t *__restrict__ sc,
                            int64_t rows_per, int *__restrict__ em) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= k) return;
    const int64_t r0 = blockIdx.y * rows_per, r1 = min(n, r0 + rows_per);
    int m = kRqZero;
    for (int64_t r = r0; r < r1; ++r) m = max(m, rq_exp(X[r * k + c], sc[r]));
    atomicMax(&em[c], m);
}

__global__ void k_rq_fixed(int64_t n, int k, const double *__restrict__ X, const int32_t *__restrict__ sc,
                           const int *__restrict__ em, int xbits, long long *__restrict__ xi) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < n * k) xi[q] = rq_fixed(X[q], sc[q / k], em[q % k], xbits);
}

// T 2^-s as double-double (T's low and high 64 bits converted apart)
__device__ __forceinline__ DD rq_dd(__int128 T) {
    const double h = (double)(long long)(T >> 64) * 18446744073709551616.0;
    const double l = (double)(unsigned long long)T;
    // |h| may be below l: an exact sum either way (TwoSum)
    const double t = h + l, z = t - h;
    // l itself may have been rounded: its error goes in with the low part
    const unsigned long long lo = (unsigned long long)T, back = l >= 18446744073709551616.0 ? 0ull : (unsigned long long)l;
    const double le = (double)(long long)(lo - back);
    return DD{t, (h - (t - z)) + (l - z) + le};
}

// Block (bx, by): rows [bx rows_per, ...) x columns [64 by, 64 by + 64).  Warp w takes rows w, w + 8, ..,
// a lane columns lane and lane + 32: y = (A x~)_i and z = (B x~)_i in 128-bit integers, then x~_i y
// and x~_i z are added to the lane's double-double numerators and denominators.  Partial
// sums: part[(bx k + c) * 4 + {num hi, num lo, den hi, den lo}].
constexpr int kRqWarps = 8;
__global__ void __launch_bounds__(32 * kRqWarps) k_rq_partial(int64_t n, const int64_t *__restrict__ rowptr,
                                                              const int32_t *__restrict__ colind,
                                                              const double *__restrict__ a, const double *__restrict__ b,
                                                              const int32_t *__restrict__ sc,
                                                              const long long *__restrict__ xi,
                                                              const int *__restrict__ em, int k, int64_t rows_per,
                                                              double *__restrict__ part) {
    __shared__ DD s_sum[kRqWarps][2][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c0 = blockIdx.y * 64;
    const int64_t r0 = blockIdx.x * rows_per, r1 = min(n, r0 + rows_per);
    const bool in[2] = {c0 + lane < k, c0 + 32 + lane < k};
    DD num[2] = {{0.0, 0.0}, {0.0, 0.0}}, den[2] = {{0.0, 0.0}, {0.0, 0.0}};
    for (int64_t i = r0 + warp; i < r1; i += kRqWarps) {
        const int64_t p0 = rowptr[i], p1 = rowptr[i + 1];
        int ea = kRqZero, eb = kRqZero;
        for (int64_t p = p0 + lane; p < p1; p += 32) {
            const int sj = -sc[colind[p]];
            ea = max(ea, rq_exp(a[p], sj));
            eb = max(eb, rq_exp(b[p], sj));
        }
        ea = __reduce_max_sync(0xffffffffu, ea);
        eb = __reduce_max_sync(0xffffffffu, eb);
        __int128 y[2] = {0, 0}, z[2] = {0, 0};
        for (int64_t q0 = p0; q0 < p1; q0 += 32) {
            const int cnt = (int)min((int64_t)32, p1 - q0);
            const bool live = lane < cnt;
            const int col = live ? colind[q0 + lane] : 0;
            const int sj = live ? -sc[col] : 0;
            const long long av = live ? rq_fixed(a[q0 + lane], sj, ea, 61) : 0;
            const long long bv = live ? rq_fixed(b[q0 + lane], sj, eb, 61) : 0;
#pragma unroll 4
            for (int e = 0; e < cnt; ++e) {
                const long long *x = xi + (int64_t)__shfl_sync(0xffffffffu, col, e) * k + c0 + lane;
                const long long ae = __shfl_sync(0xffffffffu, av, e), be = __shfl_sync(0xffffffffu, bv, e);
                const long long x0 = in[0] ? x[0] : 0, x1 = in[1] ? x[32] : 0;
                y[0] += (__int128)ae * x0;
                z[0] += (__int128)be * x0;
                y[1] += (__int128)ae * x1;
                z[1] += (__int128)be * x1;
            }
        }
        const int si = sc[i] + 1022 + 61;
        const double sa = ldexp(1.0, ea - si), sb = ldexp(1.0, eb - si);
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (in[u]) {
                const double v = (double)xi[i * k + c0 + lane + 32 * u];
                const DD ya = rq_dd(y[u]), zb = rq_dd(z[u]);
                // non-finite entries have no fixed-point form
                const double bad_a = ea == kRqNan ? __longlong_as_double(0x7ff8000000000000ll) : sa;
                const double bad_b = eb == kRqNan ? __longlong_as_double(0x7ff8000000000000ll) : sb;
                dd_add_prod(num[u], v, ya.hi * bad_a);
                dd_add_prod(num[u], v, ya.lo * bad_a);
                dd_add_prod(den[u], v, zb.hi * bad_b);
                dd_add_prod(den[u], v, zb.lo * bad_b);
            }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        s_sum[warp][0][lane + 32 * u] = num[u];
        s_sum[warp][1][lane + 32 * u] = den[u];
    }
    __syncthreads();
    const int c = threadIdx.x & 63, side = threadIdx.x >> 6;
    if (side < 2 && c0 + c < k) {
        DD t{0.0, 0.0};
        for (int w = 0; w < kRqWarps; ++w) dd_add(t, s_sum[w][side][c].hi, s_sum[w][side][c].lo);
        double *o = part + ((int64_t)blockIdx.x * k + c0 + c) * 4 + 2 * side;
        o[0] = em[c0 + c] == kRqNan ? __longlong_as_double(0x7ff8000000000000ll) : t.hi;
        o[1] = t.lo;
    }
}

// theta[c] = (sum of numerators) / (sum of denominators), summed and divided in
// double-double, rounded once
__global__ void k_rq_dd_finish(int k, int nparts, const double *__restrict__ part, double *__restrict__ theta) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= k) return;
    DD num{0.0, 0.0}, den{0.0, 0.0};
    for (int q = 0; q < nparts; ++q) {
        const double *o = part + ((int64_t)q * k + c) * 4;
        dd_add(num, o[0], o[1]);
        dd_add(den, o[2], o[3]);
    }
    const double nh = num.hi + num.lo, nl = num.lo - (nh - num.hi);
    const double dh = den.hi + den.lo, dl = den.lo - (dh - den.hi);
    const double qv = nh / dh;
    const double rem = (fma(-qv, dh, nh) + nl - qv * dl) / dh;
    theta[c] = qv + rem;
}

}  // namespace sss
