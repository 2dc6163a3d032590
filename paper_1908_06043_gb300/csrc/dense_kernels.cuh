// Dense helper kernels of the in-slice solver and the DOS sweeps (FP64).
//   Gram        G = X^T Y (Cholesky-QR Gram matrix V^T B V, projected V^T A V)
//   GEMM        Y = X Q (tall-skinny times small square: V R^-T, V Q)
//   Cholesky    G = R R^T of a small SPD matrix and R^-1
//   Jacobi      eigenpairs of small symmetric matrices by parallel-ordered cyclic Jacobi
//   Lanczos     batched dot products / updates for full re-orthogonalisation
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "grid_sync.cuh"

namespace ssd {

// ---------------------------------------------------------------- Gram G += X^T Y
// block = 32 x 32 tile of G over one chunk of rows; 256 threads, 2 x 2 outputs each, fewer where the
// matrix ends in the tile's first half (A, B outputs a thread).  A chunk of 32 rows is 16,400 clocks of
// an SM's FP64 pipe, so the rows are dealt to the whole chip, 32 a block if need be (at least 256 a
// block before: n = 5,000, k = 32 91 us, 24 now); consecutive lanes add to consecutive entries of G.
template <int A, int B>
__device__ __forceinline__ void gram_chunk(const double (*Xs)[33], const double (*Ys)[33], int tx, int ty, int rows,
                                           double (&acc)[2][2]) {
#pragma unroll 8
    for (int rr = 0; rr < rows; ++rr) {
        double x[A], y[B];
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = Xs[rr][ty + 16 * a];
#pragma unroll
        for (int b = 0; b < B; ++b) y[b] = Ys[rr][tx + 16 * b];
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int b = 0; b < B; ++b) acc[a][b] += x[a] * y[b];
    }
}
__global__ void __launch_bounds__(256) k_gram(int64_t n, const double *__restrict__ X, int64_t ldx, int k1,
                                              const double *__restrict__ Y, int64_t ldy, int k2,
                                              int64_t rows_per, int sym, double *G) {
    __shared__ double Xs[32][33], Ys[32][33];
    // sym: G is symmetric (X^T M X-type products): tiles above the diagonal only, each
    // written to both triangles
    if (sym && blockIdx.x > blockIdx.y) return;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
    const int64_t r_begin = blockIdx.z * rows_per;
    const int64_t r_end = min(n, r_begin + rows_per);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const bool a2 = i0 + 16 < k1, b2 = j0 + 16 < k2;
    double acc[2][2] = {{0, 0}, {0, 0}};
    for (int64_t r0 = r_begin; r0 < r_end; r0 += 32) {
        for (int q = tid; q < 32 * 32; q += 256) {
            int rr = q >> 5, c = q & 31;
            int64_t r = r0 + rr;
            Xs[rr][c] = (r < r_end && i0 + c < k1) ? X[r * ldx + i0 + c] : 0.0;
            Ys[rr][c] = (r < r_end && j0 + c < k2) ? Y[r * ldy + j0 + c] : 0.0;
        }
        __syncthreads();
        const int rows = (int)min((int64_t)32, r_end - r0);
        if (a2 && b2) gram_chunk<2, 2>(Xs, Ys, tx, ty, rows, acc);
        else if (a2) gram_chunk<2, 1>(Xs, Ys, tx, ty, rows, acc);
        else if (b2) gram_chunk<1, 2>(Xs, Ys, tx, ty, rows, acc);
        else gram_chunk<1, 1>(Xs, Ys, tx, ty, rows, acc);
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
            if (i < k1 && j < k2) {
                atomicAdd(&G[(int64_t)i * k2 + j], acc[a][b]);
                if (sym && blockIdx.x != blockIdx.y) atomicAdd(&G[(int64_t)j * k2 + i], acc[a][b]);
            }
        }
}

// ---------------------------------------------------------------- Y = beta Y + alpha X Q  (or X Q^T)
// block = 16 RA rows x 16 columns of Y; k1 chunks of 32 through shared memory.  Q is k1 x k2
// (ldq = k2) or, transposed, k2 x k1 (ldq = k1).  beta = 0 does not read Y.  tri: the
// effective Q (k1 x k2) is upper triangular (a lower-triangular Q used transposed), so
// chunks below column block j0's diagonal are skipped.  Bound by the FP64 pipe: RA is the largest
// that gives every SM several blocks, terms end at k1 and columns at a multiple of 16 (64 rows x 32
// columns a block and 32 terms a chunk before: n = 5,000, k = 47 73 us, 27 now).
template <int RA>
__global__ void __launch_bounds__(256) k_gemm_tall(int64_t n, const double *__restrict__ X, int64_t ldx, int k1,
                                                   const double *__restrict__ Q, int k2, int transq,
                                                   double alpha, double beta, double *__restrict__ Y,
                                                   int64_t ldy, int tri) {
    constexpr int R = 16 * RA;
    __shared__ double Xs[R][33], Qs[32][17];
    const int64_t r0 = (int64_t)blockIdx.x * R;
    const int tid = threadIdx.x, tc = tid & 15, tr = tid >> 4;   // column tc, rows tr + 16 a
    for (int64_t j0 = 16ll * blockIdx.y; j0 < k2; j0 += 16ll * gridDim.y) {
        double acc[RA];
#pragma unroll
        for (int a = 0; a < RA; ++a) acc[a] = 0.0;
        const int t_end = tri ? (int)min((int64_t)k1, j0 + 16) : k1;
        for (int t0 = 0; t0 < t_end; t0 += 32) {
            const int nt = min(32, t_end - t0);
            for (int q = tid; q < R * 32; q += 256) {
                int rr = q >> 5, c = q & 31;
                int64_t r = r0 + rr;
                Xs[rr][c] = (r < n && c < nt) ? X[r * ldx + t0 + c] : 0.0;
            }
            for (int q = tid; q < 32 * 16; q += 256) {
                const int t = transq ? q & 31 : q >> 4, c = transq ? q >> 5 : q & 15;
                double v = 0.0;
                if (t < nt && j0 + c < k2)
                    v = transq ? Q[(j0 + c) * k1 + t0 + t] : Q[(int64_t)(t0 + t) * k2 + j0 + c];
                Qs[t][c] = v;
            }
            __syncthreads();
#pragma unroll 4
            for (int t = 0; t < nt; ++t) {
                double qv = Qs[t][tc];
#pragma unroll
                for (int a = 0; a < RA; ++a) acc[a] += Xs[tr + 16 * a][t] * qv;
            }
            __syncthreads();
        }
        if (j0 + tc < k2)
#pragma unroll
            for (int a = 0; a < RA; ++a) {
                int64_t r = r0 + tr + 16 * a;
                if (r < n) {
                    double *y = Y + r * ldy + j0 + tc;
                    *y = (beta != 0.0 ? beta * *y : 0.0) + alpha * acc[a];
                }
            }
    }
}

// ---------------------------------------------------------------- small Cholesky and inverse
using ::GridBar;
using ::grid_barrier;

// G = R R^T and X = R^-1 (lower triangles, k x k row-major) in one cooperative launch, by 32-wide
// panels: the elimination of [G | I].  X must be zero on entry; G's lower triangle becomes R.  Per
// panel j
//   A  R_jj and D = R_jj^-1 (one warp of block 0, rows and then columns in registers);
//   B  R_ij = G_ij D^T for the rows below and X_j: = D X_j: for the columns before, X_jj = D;
//   C  G_il -= R_ij R_lj^T and X_ic -= R_ij X_jc for the rows below,
// with a grid barrier before B and before C; block 0 takes the next diagonal block of C and goes on
// to its A while the others do the rest.  The chain of diagonal blocks bounds it (FP64 square
// roots and 2 multiply-adds a clock on one SM); B and C are cut into items of 32 x 8 outputs to
// spread them.  k = 112: 0.67 ms as 13 launches (a one-warp diagonal kernel with a division and a
// square root a column, and an inverse of k dependent rows), 0.32 ms now.
// info[0]: first non-positive pivot + 1 (every block then leaves at its next barrier), else 0.
constexpr int CH_NB = 32;

struct CholArgs {
    double *G, *X, *D;          // D: 32 x 32 scratch
    int k;
    int *info;
    GridBar *bar;
    long long limit;
};

// R_jj and its inverse for the w x w block at column j0 (one warp; S: 32 x 33 shared scratch)
__device__ __forceinline__ void chol_diag_warp(const CholArgs &c, int j0, double (*S)[33]) {
    const int lane = threadIdx.x & 31, k = c.k, w = min(CH_NB, k - j0);
    double a[CH_NB], inv[CH_NB];
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) {
        S[t][lane] = (t < w && lane <= t) ? __ldcg(&c.G[(int64_t)(j0 + t) * k + j0 + lane]) : (t == lane ? 1.0 : 0.0);
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) a[t] = S[lane][t];       // row `lane`, columns t <= lane
    int bad = 0;
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) {
        double d = __shfl_sync(0xffffffffu, a[t], t);
        if (!(d > 0.0)) {
            if (!bad) bad = j0 + t + 1;
            d = 1.0;
        }
        inv[t] = rsqrt(d);
        a[t] *= inv[t];                                       // lane t: d / sqrt(d)
#pragma unroll
        for (int u = t + 1; u < CH_NB; ++u) a[u] -= a[t] * __shfl_sync(0xffffffffu, a[t], u);   // lanes < u: unused
    }
    __syncwarp();
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) S[lane][t] = t <= lane ? a[t] : 0.0;
    __syncwarp();
    for (int t = 0; t < w; ++t)
        if (lane <= t) c.G[(int64_t)(j0 + t) * k + j0 + lane] = S[t][lane];
    // column `lane` of the inverse, by rows
    double x[CH_NB];
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) x[t] = t == lane ? 1.0 : 0.0;
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) {
        x[t] *= inv[t];
#pragma unroll
        for (int u = t + 1; u < CH_NB; ++u) x[u] -= S[u][t] * x[t];
    }
#pragma unroll
    for (int t = 0; t < CH_NB; ++t) c.D[t * CH_NB + lane] = x[t];
    if (lane == 0 && bad) atomicCAS(c.info, 0, bad);
}

__global__ void __launch_bounds__(256) k_chol_inv(const CholArgs c) {
    __shared__ double P[32][33], Q[32][33];
    const int tid = threadIdx.x, k = c.k, nblk = (k + 31) / 32, nb = gridDim.x;
    const int r = tid >> 5, q = tid & 31;            // output (r, q) of an 8 x 32 item
    // rows [i0, i0 + m) x columns [c0, c0 + 32) of a matrix into S, zero outside k
    auto load = [&](double (*S)[33], const double *M, int i0, int m, int c0) {
        for (int e = tid; e < m * 32; e += 256)
            S[e >> 5][e & 31] = (i0 + (e >> 5) < k && c0 + (e & 31) < k) ? __ldcg(&M[(int64_t)(i0 + (e >> 5)) * k + c0 + (e & 31)]) : 0.0;
    };
    auto load_d = [&](double (*S)[33]) {
        for (int e = tid; e < 1024; e += 256) S[e >> 5][e & 31] = __ldcg(&c.D[e]);
    };
    // rows 8 sub .. of G_il -= R_i R_l^T
    auto trail_g = [&](int i, int l, int j0, int sub) {
        __syncthreads();
        load(P, c.G, 32 * i + 8 * sub, 8, j0);
        load(Q, c.G, 32 * l, 32, j0);
        __syncthreads();
        const int row = 32 * i + 8 * sub + r, col = 32 * l + q;
        if (row < k && col <= row) {
            double s = 0.0;
#pragma unroll 8
            for (int t = 0; t < 32; ++t) s += P[r][t] * Q[q][t];
            c.G[(int64_t)row * k + col] = __ldcg(&c.G[(int64_t)row * k + col]) - s;
        }
    };
    unsigned int at = 0;
    if (blockIdx.x == 0 && tid < 32) chol_diag_warp(c, 0, P);
    for (int j = 0; j < nblk; ++j) {
        const int j0 = 32 * j;
        if (!grid_barrier(c.bar, nb, c.limit, at)) return;
        if (*(volatile int *)c.info) return;          // written before the barrier: the same for every block
        // B
        const int below = nblk - 1 - j, nB = 4 * (below + j) + 1;
        for (int e = blockIdx.x; e < nB; e += nb) {
            __syncthreads();
            load_d(Q);
            if (e == nB - 1) {                         // X_jj = D
                __syncthreads();
                for (int u = tid; u < 1024; u += 256)
                    if (j0 + (u >> 5) < k && (u & 31) <= (u >> 5)) c.X[(int64_t)(j0 + (u >> 5)) * k + j0 + (u & 31)] = Q[u >> 5][u & 31];
            } else if (e < 4 * below) {                // rows of R_ij = G_ij D^T
                const int i0 = j0 + 32 * (1 + e / 4) + 8 * (e & 3);
                load(P, c.G, i0, 8, j0);
                __syncthreads();
                double s = 0.0;
#pragma unroll 8
                for (int t = 0; t < 32; ++t) s += P[r][t] * Q[q][t];
                if (i0 + r < k && j0 + q < k) c.G[(int64_t)(i0 + r) * k + j0 + q] = s;
            } else {                                   // eight columns of X_jc = D X_jc
                const int f = e - 4 * below, c0 = 8 * f;
                for (int u = tid; u < 256; u += 256)
                    P[u >> 3][u & 7] = j0 + (u >> 3) < k ? __ldcg(&c.X[(int64_t)(j0 + (u >> 3)) * k + c0 + (u & 7)]) : 0.0;
                __syncthreads();
                const int row = tid >> 3, col = tid & 7;
                double s = 0.0;
#pragma unroll 8
                for (int t = 0; t < 32; ++t) s += Q[row][t] * P[t][col];
                if (j0 + row < k) c.X[(int64_t)(j0 + row) * k + c0 + col] = s;
            }
        }
        if (below == 0) break;
        if (!grid_barrier(c.bar, nb, c.limit, at)) return;
        // C: the trailing triangle of G (its first block by block 0, which then factors it) and X
        if (blockIdx.x == 0) {
            for (int sub = 0; sub < 4; ++sub) trail_g(j + 1, j + 1, j0, sub);
            __threadfence();                           // the warp below reads them through L2
            __syncthreads();
            if (tid < 32) chol_diag_warp(c, j0 + 32, P);
        }
        const int nG = 4 * (below * (below + 1) / 2), nX = 4 * below * (j + 1);
        const int first = nb > 1 ? (int)blockIdx.x - 1 : 0, step = nb > 1 ? nb - 1 : 1;
        for (int e = first; e >= 0 && e < nG + nX; e += step) {
            if (e < nG) {
                const int pr = e >> 2;
                int i = (int)((sqrtf(8.0f * pr + 1.0f) - 1.0f) * 0.5f);
                while ((i + 1) * (i + 2) / 2 <= pr) ++i;
                while (i * (i + 1) / 2 > pr) --i;
                const int l = pr - i * (i + 1) / 2;
                if (i == 0 && l == 0) continue;        // block 0's
                trail_g(j + 1 + i, j + 1 + l, j0, e & 3);
            } else {                                   // rows of X_ic -= R_ij X_jc
                const int f = (e - nG) >> 2, i = j + 1 + f / (j + 1), cc = f % (j + 1), i0 = 32 * i + 8 * ((e - nG) & 3);
                __syncthreads();
                load(P, c.G, i0, 8, j0);
                load(Q, c.X, j0, 32, 32 * cc);
                __syncthreads();
                if (i0 + r < k) {
                    double s = 0.0;
#pragma unroll 8
                    for (int t = 0; t < 32; ++t) s += P[r][t] * Q[t][q];
                    const int64_t o = (int64_t)(i0 + r) * k + 32 * cc + q;
                    c.X[o] = __ldcg(&c.X[o]) - s;
                }
            }
        }
    }
}

// ---------------------------------------------------------------- Jacobi eigensolver
// Round r of a sweep pairs index i with partner(i) (circle method over kp = k rounded up
// to even; index kp-1 is a dummy when k is odd).  Every pair (p, q), p < q, is rotated
// by the classical Jacobi angle that annihilates H[p][q]:
//   theta = (H_qq - H_pp) / (2 H_pq), t = sign(theta) / (|theta| + sqrt(theta^2 + 1)),
//   c = 1 / sqrt(t^2 + 1), s = t c;  H' = J^T H J, V' = V J.
// t needs no more than FP32: an angle off by 1e-7 leaves 1e-7 of H[p][q], which the next sweep
// takes.  c and s are FP64 to the last bits (two Newton steps), so J stays orthogonal.  That makes a
// rotation some 15 FP64 instructions instead of two divisions and two square roots.

// pair t of round r: (p, q), p < q; q = kp - 1 >= k is the dummy of an odd k
__device__ __forceinline__ int2 jac_pair(int t, int r, int kp) {
    const int m = kp - 1;
    if (t == 0) return make_int2(r, m);
    int i = r + t, y = r - t;
    if (i >= m) i -= m;
    if (y < 0) y += m;
    return make_int2(min(i, y), max(i, y));
}

// (c, s) of the rotation of (p, q); thr: relative size below which H[p][q] is left alone
__device__ __forceinline__ double2 jac_rotation(double hpp, double hqq, double hpq, double thr) {
    if (hpq == 0.0 || hpq * hpq <= thr * thr * fabs(hpp * hqq)) return make_double2(1.0, 0.0);
    const double a = hqq - hpp, b = 2.0 * hpq;
    // theta = a / b in FP32, both scaled by the larger one's exponent
    const int ea = (int)((__double_as_longlong(a) >> 52) & 0x7ff), eb = (int)((__double_as_longlong(b) >> 52) & 0x7ff);
    const int e = max(1, min(2045, 2046 - max(ea, eb)));
    const double sc = __longlong_as_double((long long)e << 52);
    const float af = (float)(a * sc), bf = (float)(b * sc);
    const float th = af / bf;                               // bf = 0: infinite, t = 0
    const float tf = copysignf(1.0f / (fabsf(th) + sqrtf(fmaf(th, th, 1.0f))), th);
    if (!(fabsf(tf) > 0.0f)) return make_double2(1.0, 0.0);
    const double t = (double)tf, u = fma(t, t, 1.0);
    double y = (double)rsqrtf((float)u);                    // 1 <= u <= 2
    y = fma(0.5 * y, fma(-u * y, y, 1.0), y);
    y = fma(0.5 * y, fma(-u * y, y, 1.0), y);
    return make_double2(y, t * y);
}

// Parallel-ordered Jacobi on a cooperative grid, one grid barrier per round, for one or several
// matrices of the same order (group g = blockIdx.x / nb of nb blocks takes matrix g, with barrier
// g).  H is double-buffered (round r reads Ha and writes every entry of Hb, then the two swap), so
// each block can compute all of the round's rotations itself from Ha into shared memory (np x 16
// bytes of dynamic shared memory) while other blocks already write Hb; a thread loads the entries
// of its own items before it computes rotations, so a round costs one memory latency.  H is
// symmetric: items are the 2 x 2 blocks of pairs ta <= tb, written to both triangles.  acc: 2
// max_sweeps doubles a matrix (zeroed) for the per-sweep off-diagonal / total norms.  On return the
// matrix is in H (copied back from the scratch buffer H2 when the last round left it there).
// What bounds it: k - 1 rounds a sweep of barrier, load, rotation, update, store.  k = 112: 4.15 ms
// with both triangles, two divisions and two square roots a rotation and 13 blocks, 2.2 ms now;
// k = 100, four matrices: 25 ms one after the other (a single block below k = 97), 3.4 ms now.
struct JacArgs {
    double *H, *H2, *V;          // matrix g at g k^2
    int k, nb;                   // blocks per matrix
    double thr, tol;
    int max_sweeps;
    double *acc;
    GridBar *bar;
    long long limit;
};
constexpr int kJacThreads = 128;

__global__ void __launch_bounds__(kJacThreads) k_jacobi_grid(const JacArgs a) {
    extern __shared__ __align__(16) unsigned char jac_smem[];
    const int k = a.k, nb = a.nb, grp = blockIdx.x / nb, blk = blockIdx.x % nb;
    const int kp = k + (k & 1), np = kp / 2;
    double2 *s_cs = reinterpret_cast<double2 *>(jac_smem);
    const int gtid = blk * kJacThreads + threadIdx.x, gthreads = nb * kJacThreads;
    __shared__ double red_off[kJacThreads / 32], red_all[kJacThreads / 32];
    double *H = a.H + (int64_t)grp * k * k, *V = a.V + (int64_t)grp * k * k;
    double *Ha = H, *Hb = a.H2 + (int64_t)grp * k * k, *acc = a.acc + 2 * a.max_sweeps * grp;
    GridBar *bar = a.bar + grp;
    unsigned int at = 0;
    const int nH = np * (np + 1) / 2;
    auto block_of = [&](int e, int &ta, int &tb) {        // e = tb (tb + 1) / 2 + ta, ta <= tb
        tb = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
        while ((tb + 1) * (tb + 2) / 2 <= e) ++tb;
        while (tb * (tb + 1) / 2 > e) --tb;
        ta = e - tb * (tb + 1) / 2;
    };
    int ta0 = 0, tb0 = 0;
    if (gtid < nH) block_of(gtid, ta0, tb0);
    const int row0 = gtid / np, vb0 = gtid % np;          // first row pair of V
    auto load_h = [&](int2 x, int2 y, double (&h)[4]) {
        const bool rq = x.y < k, cq = y.y < k;
        h[0] = __ldcg(&Ha[(int64_t)x.x * k + y.x]);
        h[1] = cq ? __ldcg(&Ha[(int64_t)x.x * k + y.y]) : 0.0;
        h[2] = rq ? __ldcg(&Ha[(int64_t)x.y * k + y.x]) : 0.0;
        h[3] = (rq && cq) ? __ldcg(&Ha[(int64_t)x.y * k + y.y]) : 0.0;
    };
    auto turn_h = [&](int2 x, int2 y, double2 r1, double2 r2, const double (&h)[4]) {
        const bool rq = x.y < k, cq = y.y < k;
        const double u11 = r2.x * h[0] - r2.y * h[1], u12 = r2.y * h[0] + r2.x * h[1];
        const double u21 = r2.x * h[2] - r2.y * h[3], u22 = r2.y * h[2] + r2.x * h[3];
        const double b11 = r1.x * u11 - r1.y * u21, b21 = r1.y * u11 + r1.x * u21;
        double b12 = r1.x * u12 - r1.y * u22;
        const double b22 = r1.y * u12 + r1.x * u22;
        if (x.x == y.x) b12 = b21;                        // a diagonal block stays symmetric
        Hb[(int64_t)x.x * k + y.x] = b11;
        Hb[(int64_t)y.x * k + x.x] = b11;
        if (cq) { Hb[(int64_t)x.x * k + y.y] = b12; Hb[(int64_t)y.y * k + x.x] = b12; }
        if (rq) { Hb[(int64_t)x.y * k + y.x] = b21; Hb[(int64_t)y.x * k + x.y] = b21; }
        if (rq && cq) { Hb[(int64_t)x.y * k + y.y] = b22; Hb[(int64_t)y.y * k + x.y] = b22; }
    };
    int sweep = 0;
    for (; sweep < a.max_sweeps; ++sweep) {
        double off = 0.0, all = 0.0;
        for (int64_t q = gtid; q < (int64_t)k * k; q += gthreads) {
            const double h = __ldcg(&Ha[q]), v = h * h;
            all += v;
            if (q / k != q % k) off += v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_down_sync(0xffffffffu, off, o);
            all += __shfl_down_sync(0xffffffffu, all, o);
        }
        if ((threadIdx.x & 31) == 0) { red_off[threadIdx.x >> 5] = off; red_all[threadIdx.x >> 5] = all; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double o2 = 0.0, a2 = 0.0;
            for (int w = 0; w < kJacThreads / 32; ++w) { o2 += red_off[w]; a2 += red_all[w]; }
            atomicAdd(&acc[2 * sweep], o2);
            atomicAdd(&acc[2 * sweep + 1], a2);
        }
        if (!grid_barrier(bar, nb, a.limit, at)) return;
        const double o2 = *(volatile double *)&acc[2 * sweep], a2 = *(volatile double *)&acc[2 * sweep + 1];
        if (o2 <= a.tol * a.tol * a2) break;
        for (int r = 0; r < kp - 1; ++r) {
            // this thread's first items, then the round's rotations
            double h[4], v0 = 0.0, v1 = 0.0;
            const int2 x0 = jac_pair(ta0, r, kp), y0 = jac_pair(tb0, r, kp), z0 = jac_pair(vb0, r, kp);
            if (gtid < nH) load_h(x0, y0, h);
            if (row0 < k && z0.y < k) {
                v0 = __ldcg(&V[(int64_t)row0 * k + z0.x]);
                v1 = __ldcg(&V[(int64_t)row0 * k + z0.y]);
            }
            for (int t = threadIdx.x; t < np; t += kJacThreads) {
                const int2 pq = jac_pair(t, r, kp);
                s_cs[t] = pq.y < k ? jac_rotation(__ldcg(&Ha[(int64_t)pq.x * k + pq.x]), __ldcg(&Ha[(int64_t)pq.y * k + pq.y]),
                                                  __ldcg(&Ha[(int64_t)pq.x * k + pq.y]), a.thr)
                                   : make_double2(1.0, 0.0);
            }
            __syncthreads();
            // Hb = J^T Ha J, every 2 x 2 block written
            if (gtid < nH) turn_h(x0, y0, s_cs[ta0], s_cs[tb0], h);
            for (int e = gtid + gthreads; e < nH; e += gthreads) {
                int ta, tb;
                block_of(e, ta, tb);
                const int2 x = jac_pair(ta, r, kp), y = jac_pair(tb, r, kp);
                load_h(x, y, h);
                turn_h(x, y, s_cs[ta], s_cs[tb], h);
            }
            // V = V J (each entry updated by exactly one thread per round)
            if (row0 < k && z0.y < k) {
                const double2 c = s_cs[vb0];
                V[(int64_t)row0 * k + z0.x] = c.x * v0 - c.y * v1;
                V[(int64_t)row0 * k + z0.y] = c.y * v0 + c.x * v1;
            }
            for (int e = gtid + gthreads; e < k * np; e += gthreads) {
                const int row = e / np, tb = e - row * np;
                const int2 z = jac_pair(tb, r, kp);
                const double2 c = s_cs[tb];
                if (z.y >= k || c.y == 0.0) continue;
                double *vr = V + (int64_t)row * k;
                const double vp = __ldcg(&vr[z.x]), vq = __ldcg(&vr[z.y]);
                vr[z.x] = c.x * vp - c.y * vq;
                vr[z.y] = c.y * vp + c.x * vq;
            }
            if (!grid_barrier(bar, nb, a.limit, at)) return;
            double *t = Ha;
            Ha = Hb;
            Hb = t;
        }
    }
    if (Ha != H)
        for (int64_t q = gtid; q < (int64_t)k * k; q += gthreads) H[q] = __ldcg(&Ha[q]);
}

// ascending eigenvalues with their eigenvector columns: rank by (value, index).  Block (bx, g): matrix
// g, rows 32 bx .. + 31 of Q; every block ranks all values itself.
__global__ void __launch_bounds__(256) k_eig_sort(const double *__restrict__ H, const double *__restrict__ V, int k,
                                                  double *__restrict__ evals, double *__restrict__ Q) {
    extern __shared__ __align__(16) double s_val[];            // k values, then their ranks
    int *rank = reinterpret_cast<int *>(s_val + k);
    const int64_t off = (int64_t)blockIdx.y * k * k;
    for (int i = threadIdx.x; i < k; i += 256) s_val[i] = H[off + (int64_t)i * k + i];
    __syncthreads();
    for (int i = threadIdx.x; i < k; i += 256) {
        const double li = s_val[i];
        int r = 0;
        for (int j = 0; j < k; ++j) {
            const double lj = s_val[j];
            if (lj < li || (lj == li && j < i)) ++r;
        }
        rank[i] = r;
        if (blockIdx.x == 0) evals[(int64_t)blockIdx.y * k + r] = li;
    }
    __syncthreads();
    const int r0 = blockIdx.x * 32, r1 = min(k, r0 + 32);
    for (int e = threadIdx.x; e < (r1 - r0) * k; e += 256) {
        const int row = r0 + e / k, i = e % k;
        Q[off + (int64_t)row * k + rank[i]] = V[off + (int64_t)row * k + i];
    }
}

// copy an n x k block between leading dimensions
__global__ void k_copy_cols(int64_t n, int k, const double *__restrict__ X, int64_t ldx, double *__restrict__ Y,
                            int64_t ldy) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= n * k) return;
    const int64_t r = q / k;
    const int c = (int)(q - r * k);
    Y[r * ldy + c] = X[r * ldx + c];
}

__global__ void k_set_identity(double *V, int k) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q < (int64_t)k * k) V[(int64_t)blockIdx.y * k * k + q] = (q / k == q % k) ? 1.0 : 0.0;
}

// ---------------------------------------------------------------- column reductions
// out[c] += sum of acc over the block's threads tid = c mod nv; 256 threads, nv a power of two.
// Within warps by shuffles: as one thread a column over 256 / nv values it was most of such a launch.
__device__ __forceinline__ void column_sums(double acc, int nv, double *s, double *out) {
    const int tid = threadIdx.x, step = max(nv, 32);
    for (int o = 16; o >= nv; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    s[tid] = acc;
    __syncthreads();
    if (tid < nv) {
        double v = 0.0;
        for (int t = tid; t < 256; t += step) v += s[t];
        atomicAdd(&out[tid], v);
    }
}
// out[c] += sum_r X[r][c] * Y[r][c]
__global__ void k_col_dot(int64_t n, int k, const double *__restrict__ X, const double *__restrict__ Y,
                          double *out) {
    // requires 256 % k == 0 so that each thread keeps one column
    __shared__ double s[256];
    const int tid = threadIdx.x;
    double acc = 0.0;
    const int64_t tot = n * k;
    for (int64_t q = blockIdx.x * 256ll + tid; q < tot; q += (int64_t)gridDim.x * 256)
        acc += X[q] * Y[q];
    column_sums(acc, k, s, out);
}

// out[c] += sum_r X[r][c]^2 for any k (block per row chunk)
__global__ void k_col_sumsq(int64_t n, int k, const double *__restrict__ X, int64_t rows_per,
                            double *out) {
    const int64_t r0 = blockIdx.y * rows_per, r1 = min(n, r0 + rows_per);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < k; c += gridDim.x * blockDim.x) {
        double acc = 0.0;
        for (int64_t r = r0; r < r1; ++r) {
            double v = X[r * k + c];
            acc += v * v;
        }
        atomicAdd(&out[c], acc);
    }
}

// rr[c] += sum_r (AX[r][c] - theta[c] BX[r][c])^2 and xx[c] += sum_r X[r][c]^2: residual and vector
// norms, squared, of the rows of one block
__global__ void k_resid_sumsq(int64_t n, int k, const double *__restrict__ AX, const double *__restrict__ BX,
                              const double *__restrict__ X, const double *__restrict__ theta, int64_t rows_per,
                              double *rr, double *xx) {
    const int64_t r0 = blockIdx.y * rows_per, r1 = min(n, r0 + rows_per);
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= k) return;
    const double th = theta[c];
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (int64_t r = r0; r < r1; ++r) {
        const double v = AX[r * k + c] - th * BX[r * k + c], x = X[r * k + c];
        a += v * v;
        b += x * x;
    }
    atomicAdd(&rr[c], a);
    atomicAdd(&xx[c], b);
}

// resid[c] = sqrt(rr[c]) / (normA * sqrt(xx[c]))
__global__ void k_resid_finish(int k, const double *__restrict__ rr, const double *__restrict__ xx,
                               double normA, double *__restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < k) out[c] = sqrt(rr[c]) / (normA * sqrt(xx[c]));
}

__global__ void k_neg_scale(int k, const double *__restrict__ x, double *__restrict__ y) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < k) y[c] = -x[c];
}

// ---------------------------------------------------------------- Lanczos helpers
// h[i][c] = sum_r Q_i[r][c] w[r][c], i < j; grid (j, chunks); 256 % nv == 0
__global__ void __launch_bounds__(256) k_lz_dots(const double *__restrict__ Qb, int64_t n, int nv, int j,
                          const double *__restrict__ w, int64_t per, double *h) {
    __shared__ double s[256];
    const int i = blockIdx.x;
    const int tid = threadIdx.x;
    const int64_t tot = n * nv;
    const int64_t e0 = blockIdx.y * per, e1 = min(tot, e0 + per);
    const double *q = Qb + (int64_t)i * tot;
    double acc = 0.0;
#pragma unroll 8
    for (int64_t e = e0 + tid; e < e1; e += 256) acc += q[e] * w[e];
    column_sums(acc, nv, s, h + (int64_t)i * nv);
}
// Re-orthogonalisation, N = 2,688, 4 vectors, 100 steps: 109 us a step with one block a vector in the
// dots, one thread an entry over all vectors here and one launch an array; 57 us now, of which most is
// launches and the L2's latency.
// w -= sum_i X_i h_i (blockIdx.y = 0) and bw -= sum_i BX_i h_i (1): block = 32 entries, the vectors
// dealt to 8 warps
__global__ void __launch_bounds__(256) k_lz_sub(const double *__restrict__ X, const double *__restrict__ BX, int64_t n,
                                                int nv, int j, const double *__restrict__ h, double *w, double *bw) {
    __shared__ double s[8][33];
    const int64_t tot = n * nv, e = blockIdx.x * 32ll + (threadIdx.x & 31);
    const int part = threadIdx.x >> 5, lane = threadIdx.x & 31, c = (int)(e % nv);
    const double *Q = blockIdx.y ? BX : X;
    double acc = 0.0;
    if (e < tot)
#pragma unroll 4
        for (int i = part; i < j; i += 8) acc += Q[(int64_t)i * tot + e] * h[(int64_t)i * nv + c];
    s[part][lane] = acc;
    __syncthreads();
    if (part == 0 && e < tot) {
        double v = 0.0;
#pragma unroll
        for (int p = 0; p < 8; ++p) v += s[p][lane];
        double *o = blockIdx.y ? bw : w;
        o[e] -= v;
    }
}
__global__ void k_lz_three_term(int64_t n, int nv, const double *__restrict__ q,
                                const double *__restrict__ qp, const double *__restrict__ alpha,
                                const double *__restrict__ beta_prev, double *w) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= n * nv) return;
    const int c = (int)(e % nv);
    double v = w[e] - alpha[c] * q[e];
    if (beta_prev) v -= beta_prev[c] * qp[e];
    w[e] = v;
}

// x = w / beta and bx = bw / beta (blockIdx.y) with beta = sqrt(nrm2), 0 for beta = 0; one root and
// reciprocal a column, the quotient corrected to about its last bit
__global__ void __launch_bounds__(256) k_lz_normalize(int64_t n, int nv, const double *__restrict__ w,
                               const double *__restrict__ bw, const double *__restrict__ nrm2, double *__restrict__ beta,
                               double *__restrict__ x, double *__restrict__ bx) {
    __shared__ double s_b[256], s_r[256];
    const int64_t e = blockIdx.x * 256ll + threadIdx.x;
    if (threadIdx.x < nv) {
        const double b = sqrt(nrm2[threadIdx.x]);
        s_b[threadIdx.x] = b;
        s_r[threadIdx.x] = 1.0 / b;
        if (blockIdx.x == 0 && blockIdx.y == 0) beta[threadIdx.x] = b;
    }
    __syncthreads();
    if (e >= n * nv) return;
    const int c = (int)(e % nv);
    const double b = s_b[c], r = s_r[c], v = (blockIdx.y ? bw : w)[e];
    double q = v * r;
    q += r * fma(-q, b, v);
    if (!isfinite(q)) q = v / b;
    (blockIdx.y ? bx : x)[e] = b > 0.0 ? q : 0.0;
}
__global__ void k_lz_tridiag(const double *__restrict__ alpha, const double *__restrict__ beta,
                             int nv, int c, int m, double *T) {
    const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (q >= (int64_t)m * m) return;
    const int i = (int)(q / m), j = (int)(q % m);
    double v = 0.0;
    if (i == j) v = alpha[(int64_t)i * nv + c];
    else if (j == i + 1) v = beta[(int64_t)i * nv + c];
    else if (i == j + 1) v = beta[(int64_t)j * nv + c];
    T[q] = v;
}

}  // namespace ssd
