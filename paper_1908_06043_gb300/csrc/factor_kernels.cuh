// Numeric multifrontal LDL^T kernels (Alg. 2 step 2: (L, D) <- LDL^T of A - sigma B).
//
// A front is a dense column-major m x m block in the level workspace; only its lower
// triangle is meaningful.  Its first ncol columns are eliminated in panels of width
// w <= 64; each panel step is
//   K2 diag:  FP64 Bunch-Kaufman on the w x w diagonal block, pivots restricted to the
//             block: P F11 P^T = L D L^T.  Writes L^-1, D, the local pivot order and
//             the transform Mt = P^T L^-T D^-1, and counts the inertia of D.
//   K4 panel: L21 = F21 Mt (in place) and W = L21 D (scratch), 16- to 64-row tiles.
//   K3 Schur: F22 -= L21 W^T on the lower-triangular 64 x 64 tiles of the trailing front.
// Before a level's steps its fronts are zeroed, the stored entries of A - sigma B are
// scattered in (assembly) and the children's contribution blocks are added from the pool
// (extend-add, one pass per child slot so that no two blocks of a pass write the same
// parent entry).  After them the fronts' panel columns go to L storage and their trailing
// blocks to the pool (store), so the workspace holds one level at a time.
// Every kernel is batched over shifts with blockIdx.y.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace ssk {

constexpr int NB = 64;     // panel width
constexpr int TR = 64;     // row tile of the panel transform / Schur update
template <typename T, int RA> constexpr size_t panel_smem() { return NB * (NB + 1 + 2 * (16 * RA + 1)) * sizeof(T); }
template <typename T> constexpr size_t schur_smem() { return 2 * NB * (TR + 1) * sizeof(T); }

template <typename T>
struct ShiftPtrs {
    const double *a, *b;            // pencil values on the pattern (caller-owned)
    T *ws;                          // level workspace (fronts of the level being factored)
    T *cb;                          // contribution-block pool
    T *lst;                         // L storage (null: inertia only, nothing kept)
    double *linv;                   // npanels * NB * NB, row-major L^-1 of each panel
    double *dblk;                   // npanels * 2 * NB: D diagonal then sub-diagonal
    int32_t *piv;                   // npanels * NB
    T *mt;                          // mt_max * NB * NB
    T *wbuf;                        // wbuf_max
    unsigned char *sl;              // operand slices of the tensor-core Schur update
    int32_t *ex;                    // their row exponents
    unsigned long long *counts;     // [neg, zero, pos, tiny, min_pivot_bits, n2x2, max_abs_l_bits, timeouts]
    const double *seg_sigma;        // several pencils in one block-diagonal pattern: the shift
    const int32_t *eseg;            // of each pencil (seg_sigma) and the pencil of each stored
                                    // entry (eseg); null for one pencil (sigma)
    double sigma;
    double tiny_thr;                // pivots below this are flagged
    double norm;                    // ||A - sigma B||_1 bound (for min-pivot ratio)
};

// ---------------------------------------------------------------- assembly
template <typename T>
__global__ void k_assemble(int64_t count, const int32_t *__restrict__ asm_e,
                           const int64_t *__restrict__ asm_dest, const ShiftPtrs<T> *sp) {
    const ShiftPtrs<T> s = sp[blockIdx.y];
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < count;
         q += (int64_t)gridDim.x * blockDim.x) {
        int32_t e = asm_e[q];
        const double sg = s.eseg ? s.seg_sigma[s.eseg[e]] : s.sigma;
        s.ws[asm_dest[q]] = (T)(s.a[e] - sg * s.b[e]);
    }
}

// Inertia of D per pencil of a block-diagonal pattern: every panel's 1x1 and 2x2 pivots
// (the classification of k_diag_bk) counted for the pencil its rows belong to.  seg:
// pencil of each original row; perm: permuted -> original row; out: n_seg x 4
// (neg, zero, pos, tiny).
__global__ void k_segment_inertia(int32_t npan, const PanelDesc *__restrict__ panels,
                                  const double *__restrict__ dblk, const int32_t *__restrict__ perm,
                                  const int32_t *__restrict__ seg, double tiny_thr,
                                  unsigned long long *__restrict__ out) {
    const int p = blockIdx.x;
    if (p >= npan) return;
    const PanelDesc pd = panels[p];
    const int i = threadIdx.x;
    if (i >= pd.w) return;
    const double *dd = dblk + (int64_t)p * 2 * NB, *de = dd + NB;
    unsigned long long *o = out + 4ll * seg[perm[pd.g0]];
    if (i > 0 && de[i - 1] != 0.0) return;                 // second row of a 2x2 block
    if (de[i] != 0.0) {                                     // 2x2 block (i, i+1)
        const double a = dd[i], b = de[i], c = dd[i + 1], det = a * c - b * b, tr = a + c;
        if (det < 0) { atomicAdd(&o[0], 1ull); atomicAdd(&o[2], 1ull); }
        else if (det > 0) atomicAdd(&o[tr > 0 ? 2 : 0], 2ull);
        else { atomicAdd(&o[1], 1ull); atomicAdd(&o[tr > 0 ? 2 : (tr < 0 ? 0 : 1)], 1ull); }
        const double emax = fabs(0.5 * tr) + sqrt(0.25 * (a - c) * (a - c) + b * b);
        const double emin = emax > 0 ? fabs(det) / emax : 0.0;
        if (emin < tiny_thr) atomicAdd(&o[3], 1ull);
    } else {
        const double d = dd[i];
        atomicAdd(&o[d < 0 ? 0 : (d > 0 ? 2 : 1)], 1ull);
        if (fabs(d) < tiny_thr) atomicAdd(&o[3], 1ull);
    }
}

// ---------------------------------------------------------------- extend-add
// One block per contribution column: parent[rel[i], rel[j]] += cb[i, j], i >= j.  A block
// in the pool is its lower triangle packed by columns: column j (rows j .. nr-1) starts
// at j (2 nr - j + 1) / 2.
template <typename T>
__global__ void k_extend_add(const ExtendTask *__restrict__ tasks, int32_t ntask,
                             const int32_t *__restrict__ relmap, const ShiftPtrs<T> *sp) {
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const int32_t col = blockIdx.x;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].col_pre <= col) lo = mid; else hi = mid - 1;
    }
    const ExtendTask t = tasks[lo];
    const int32_t j = col - t.col_pre;
    const int32_t nr = t.child_m - t.child_ncol;
    const int32_t *rel = relmap + t.rel_off;
    const T *cc = s.cb + t.child_off + (int64_t)j * (2 * (int64_t)nr - j - 1) / 2;   // cc[i]: row i >= j
    T *pc = s.ws + t.parent_off + (int64_t)rel[j] * t.parent_m;
    for (int32_t i = j + threadIdx.x; i < nr; i += blockDim.x) pc[rel[i]] += cc[i];
}

// ---------------------------------------------------------------- store
// One block per front column of a level: column c < ncol to L storage (all m rows),
// column ncol + j to the contribution-block pool (rows j .. nr-1, packed lower triangle).
template <typename T>
__global__ void k_level_store(const StoreTask *__restrict__ tasks, int32_t ntask, const ShiftPtrs<T> *sp) {
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const int32_t col = blockIdx.x;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].col_pre <= col) lo = mid; else hi = mid - 1;
    }
    const StoreTask t = tasks[lo];
    const int32_t c = col - t.col_pre;
    const T *src = s.ws + t.ws_off + (int64_t)c * t.m;
    if (c < t.ncol) {
        if (!s.lst) return;
        T *dst = s.lst + t.l_off + (int64_t)c * t.m;
        for (int32_t i = threadIdx.x; i < t.m; i += blockDim.x) dst[i] = src[i];
    } else {
        const int32_t j = c - t.ncol, nr = t.m - t.ncol;
        T *dst = s.cb + t.cb_off + (int64_t)j * (2 * (int64_t)nr - j - 1) / 2;    // dst[i]: row i >= j
        src += t.ncol;
        for (int32_t i = j + threadIdx.x; i < nr; i += blockDim.x) dst[i] = src[i];
    }
}

// ---------------------------------------------------------------- K2: diagonal block
// One block per (front, shift).  FP64 runs at 2 multiply-adds a clock here, on one SM, so the
// block does only the lower triangle's (w^3 / 6) and the inverse's (w^3 / 6), with one multiply-add
// each and no division in a loop; pivots are compared as integers (|x| orders like its bits).
// Per column one block barrier: warp 0 runs one column ahead -- it updates column k + 1, finds
// its largest entry and, when the diagonal passes the 1x1 test, forms 1 / d and that column of L,
// while warps 1-7 update the rest in 8 x 4 patches.  Only where the test fails do the second
// search, the symmetric swap or the 2x2 pivot take barriers of their own.  N = 16,384, 164 steps:
// 330 us a step with the full square updated by three FP64 operations an entry behind a
// whole-block barrier per action and a serial column-per-thread inverse; 118 us now.
constexpr int DLD = NB + 4;        // row stride: 8 x 4 patches touch every shared-memory bank once
constexpr size_t kDiagSmem = 2 * NB * DLD * sizeof(double);

__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ double from_bits(unsigned long long b) { return __longlong_as_double((long long)b); }

// largest key over the warp and the smallest index holding it
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key, int &idx) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    idx = (int)__reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? (unsigned)idx : 0x7fffffffu);
    return ((unsigned long long)mh << 32) | ml;
}

template <typename T>
__global__ void __launch_bounds__(256) k_diag_bk(const StepTask *__restrict__ tasks, const ShiftPtrs<T> *sp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *A = reinterpret_cast<double *>(smem_raw);       // lower triangle, entry (i, j) at i DLD + j
    double *L = A + NB * DLD;                                // strict lower part of L
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const StepTask tk = tasks[blockIdx.x];
    const int w = tk.w, m = tk.m, k0 = tk.k0;
    __shared__ int perm[NB];
    __shared__ double dd[NB], de[NB], p0[NB], p1[NB];
    __shared__ int s_kind, s_r, s_fast[2];
    __shared__ unsigned long long c_neg, c_zero, c_pos, c_tiny, c_2x2;
    __shared__ double s_minpiv;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T *F = s.ws + tk.front_off;

    for (int q = tid; q < NB * NB; q += 256) {
        const int j = q / NB, i = q % NB;                    // column j, row i (coalesced on i)
        if (i >= j && i < w) A[i * DLD + j] = (double)F[(int64_t)(k0 + j) * m + (k0 + i)];
    }
    for (int q = tid; q < NB * DLD; q += 256) L[q] = 0.0;
    if (tid < NB) { perm[tid] = tid; dd[tid] = 0.0; de[tid] = 0.0; }
    if (tid == 0) {
        c_neg = c_zero = c_pos = c_tiny = c_2x2 = 0;
        s_minpiv = 1e300;
        s_fast[0] = 0;
    }
    __syncthreads();

    const double alpha = 0.6403882032022076;   // (1 + sqrt(17)) / 8
    // column k of L for a 1x1 pivot d at k (warp 0)
    auto scale_column = [&](int k, double d, double v1, double v2) {
        const double inv = d != 0.0 ? 1.0 / d : 0.0;
        const int i1 = k + 1 + lane, i2 = i1 + 32;
        if (i1 < w) L[i1 * DLD + k] = v1 * inv;
        if (i2 < w) L[i2 * DLD + k] = v2 * inv;
    };
    // A(i, j) -= x(i) y(j) [+ x2(i) y2(j)] on the trailing triangle from row / column b0, in 8 x 4
    // patches dealt to warps first, first + 1, ..; x = column c of L, y = column c of A
    auto update = [&](int b0, int c, bool two, int first, int nwarp) {
        const int n2 = w - b0, npr = (n2 + 7) >> 3, np = npr * (npr + 1);
        int pr = 0;
        for (int p = warp - first; p < np; p += nwarp) {
            while (p >= (pr + 1) * (pr + 2)) ++pr;
            const int i = b0 + 8 * pr + (lane >> 2), j = b0 + 4 * (p - pr * (pr + 1)) + (lane & 3);
            if (i < w && j <= i) {
                double v = A[i * DLD + j];
                v -= L[i * DLD + c] * A[j * DLD + c];
                if (two) v -= L[i * DLD + c + 1] * A[j * DLD + c + 1];
                A[i * DLD + j] = v;
            }
        }
    };
    int k = 0;
    for (int it = 0; k < w; ++it) {
        int kind = 1;
        if (!s_fast[it & 1]) {
            // the pivot of column k: Bunch-Kaufman's test restricted to the block
            if (warp == 0) {
                unsigned long long key = 0;
                int r = k;
                const int i1 = k + 1 + lane, i2 = i1 + 32;
                const double v1 = i1 < w ? A[i1 * DLD + k] : 0.0, v2 = i2 < w ? A[i2 * DLD + k] : 0.0;
                if (i1 < w) { key = abs_bits(v1); r = i1; }
                if (i2 < w && abs_bits(v2) > key) { key = abs_bits(v2); r = i2; }
                if (k + 1 < w) key = warp_max_key(key, r);
                const double lam = from_bits(key), d = A[k * DLD + k], akk = fabs(d);
                int kd = 1;                          // 1: 1x1 at k; 2: 1x1 with swap k<->r; 3: 2x2 (k+1<->r)
                if (akk < alpha * lam) {
                    unsigned long long ks = 0;
                    int dummy = 0;
                    for (int j = k + lane; j < w; j += 32) {
                        if (j == r) continue;
                        const unsigned long long kj = abs_bits(j < r ? A[r * DLD + j] : A[j * DLD + r]);
                        if (kj > ks) ks = kj;
                    }
                    const double sig = from_bits(warp_max_key(ks, dummy));
                    if (akk * sig >= alpha * lam * lam) kd = 1;
                    else if (fabs(A[r * DLD + r]) >= alpha * sig) kd = 2;
                    else kd = 3;
                }
                if (kd == 1) scale_column(k, d, v1, v2);
                if (lane == 0) { s_kind = kd; s_r = r; }
            }
            __syncthreads();
            kind = s_kind;
            const int r = s_r;
            if (kind >= 2) {
                const int a = (kind == 2) ? k : k + 1;
                if (a != r) {                        // symmetric swap a <-> r of A, row swap of L
                    if (tid < w && tid != r) {
                        const int j = tid;
                        double *x, *y;
                        if (j < k) { x = &L[a * DLD + j]; y = &L[r * DLD + j]; }
                        else if (j < a) { x = &A[a * DLD + j]; y = &A[r * DLD + j]; }
                        else if (j == a) { x = &A[a * DLD + a]; y = &A[r * DLD + r]; }
                        else if (j < r) { x = &A[j * DLD + a]; y = &A[r * DLD + j]; }
                        else { x = &A[j * DLD + a]; y = &A[j * DLD + r]; }
                        const double t = *x;
                        *x = *y;
                        *y = t;
                    }
                    if (tid == 0) { const int t = perm[a]; perm[a] = perm[r]; perm[r] = t; }
                    __syncthreads();
                }
                if (kind == 2) {
                    if (warp == 0) {
                        const int i1 = k + 1 + lane, i2 = i1 + 32;
                        scale_column(k, A[k * DLD + k], i1 < w ? A[i1 * DLD + k] : 0.0, i2 < w ? A[i2 * DLD + k] : 0.0);
                    }
                    __syncthreads();
                }
            }
        }
        if (kind <= 2) {
            if (warp == 0) {
                // column k + 1 ahead of the others: update, search, 1x1 test, its column of L
                int fast = 0;
                if (k + 1 < w) {
                    const double c = A[(k + 1) * DLD + k];
                    const int i0 = k + 1 + lane, i1 = i0 + 32;
                    double v0 = 0.0, v1 = 0.0;
                    if (i0 < w) { v0 = A[i0 * DLD + k + 1] - L[i0 * DLD + k] * c; A[i0 * DLD + k + 1] = v0; }
                    if (i1 < w) { v1 = A[i1 * DLD + k + 1] - L[i1 * DLD + k] * c; A[i1 * DLD + k + 1] = v1; }
                    const double d = __shfl_sync(0xffffffffu, v0, 0);
                    unsigned long long key = lane > 0 ? abs_bits(v0) : 0;
                    if (abs_bits(v1) > key) key = abs_bits(v1);
                    int dummy = 0;
                    key = warp_max_key(key, dummy);
                    const double inv = d != 0.0 ? 1.0 / d : 0.0;
                    fast = !(fabs(d) < alpha * from_bits(key));
                    if (fast) {
                        if (lane > 0 && i0 < w) L[i0 * DLD + k + 1] = v0 * inv;
                        if (i1 < w) L[i1 * DLD + k + 1] = v1 * inv;
                    }
                }
                if (lane == 0) s_fast[(it + 1) & 1] = fast;
            } else {
                if (tid == 32) {
                    const double d = A[k * DLD + k], ad = fabs(d);
                    dd[k] = d;
                    if (d < 0) c_neg++; else if (d > 0) c_pos++; else c_zero++;
                    if (ad < s.tiny_thr) c_tiny++;
                    if (ad < s_minpiv) s_minpiv = ad;
                }
                update(k + 2, k, false, 1, 7);
            }
            __syncthreads();
            k += 1;
        } else {
            const double a = A[k * DLD + k], b = A[(k + 1) * DLD + k], c = A[(k + 1) * DLD + k + 1];
            const double det = a * c - b * b;
            if (tid == 32) {
                dd[k] = a; dd[k + 1] = c; de[k] = b; de[k + 1] = 0.0;
                c_2x2++;
                double tr = a + c;
                if (det < 0) { c_neg++; c_pos++; }
                else if (det > 0) { if (tr > 0) c_pos += 2; else c_neg += 2; }
                else { c_zero++; if (tr > 0) c_pos++; else if (tr < 0) c_neg++; else c_zero++; }
                double emax = fabs(0.5 * tr) + sqrt(0.25 * (a - c) * (a - c) + b * b);
                double emin = emax > 0 ? fabs(det) / emax : 0.0;
                if (emin < s.tiny_thr) c_tiny++;
                if (emin < s_minpiv) s_minpiv = emin;
            }
            const int i = k + 2 + tid;
            if (i < w) {
                const double id = 1.0 / det, ci0 = A[i * DLD + k], ci1 = A[i * DLD + k + 1];
                L[i * DLD + k] = (c * ci0 - b * ci1) * id;
                L[i * DLD + k + 1] = (-b * ci0 + a * ci1) * id;
            }
            if (tid == 0) s_fast[(it + 1) & 1] = 0;
            __syncthreads();
            update(k + 2, k, true, 0, 8);
            __syncthreads();
            k += 2;
        }
    }
    // X = L^-1 in A's place, by 16 x 16 diagonal blocks and two levels of
    // X21 = -X22 (L21 X11); the products L21 X11 rest in blocks above the diagonal meanwhile
    double *X = A;
    if (tid < NB) {
        const int b = tid & ~15, jl = tid & 15;
        double x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = i == jl ? 1.0 : 0.0;
#pragma unroll
        for (int t = 0; t < 15; ++t)
#pragma unroll
            for (int i = t + 1; i < 16; ++i) x[i] -= L[(b + i) * DLD + b + t] * x[t];
#pragma unroll
        for (int i = 0; i < 16; ++i) X[(b + i) * DLD + tid] = x[i];
    } else {
        // constants of D^-1: column j of L^-T D^-1 is p0 X(j, :) + p1 X(j +- 1, :)
        const int j = tid - NB;
        if (j < w) {
            const bool first2 = de[j] != 0.0, second2 = j > 0 && de[j - 1] != 0.0;
            if (first2 || second2) {
                const int f = first2 ? j : j - 1;
                const double a = dd[f], b = de[f], c = dd[f + 1], det = a * c - b * b;
                p0[j] = (first2 ? c : a) / det;
                p1[j] = -b / det;
            } else {
                p0[j] = dd[j] != 0.0 ? 1.0 / dd[j] : 0.0;
                p1[j] = 0.0;
            }
        }
    }
    __syncthreads();
    {
        const int h = lane & 15, C = 32 * (lane >> 4), R = C + 16;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = warp + 8 * u;
            double acc = 0.0;
            for (int t = j; t < 16; ++t) acc += L[(R + h) * DLD + C + t] * X[(C + t) * DLD + C + j];
            X[(C + h) * DLD + R + j] = acc;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = warp + 8 * u;
            double acc = 0.0;
            for (int t = 0; t <= i; ++t) acc += X[(R + i) * DLD + R + t] * X[(C + t) * DLD + R + h];
            X[(R + i) * DLD + C + h] = -acc;
        }
        __syncthreads();
        if (w > 32) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = warp + 8 * u;
                double acc = 0.0;
                for (int t = j; t < 32; ++t) acc += L[(32 + lane) * DLD + t] * X[t * DLD + j];
                X[lane * DLD + 32 + j] = acc;
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = warp + 8 * u;
                double acc = 0.0;
                for (int t = 0; t <= i; ++t) acc += X[(32 + i) * DLD + 32 + t] * X[t * DLD + 32 + lane];
                X[(32 + i) * DLD + lane] = -acc;
            }
            __syncthreads();
        }
    }
    const int p = tk.panel;
    double *linv = s.linv + (int64_t)p * NB * NB;
    unsigned long long lmax = 0;                 // largest |L| entry (element growth diagnostic)
    for (int q = tid; q < NB * NB; q += 256) {
        const int i = q / NB, j = q % NB;
        linv[q] = (i < w && j <= i) ? X[i * DLD + j] : 0.0;
        if (i > j) lmax = max(lmax, abs_bits(L[i * DLD + j]));
    }
    if (tid < NB) {
        s.dblk[(int64_t)p * 2 * NB + tid] = tid < w ? dd[tid] : 0.0;
        s.dblk[(int64_t)p * 2 * NB + NB + tid] = tid < w ? de[tid] : 0.0;
        s.piv[(int64_t)p * NB + tid] = tid < w ? perm[tid] : tid;
    }
    // Mt[perm[i]][j] = sum_{t in block(j)} Li[t][i] Dinv[t][j]
    T *mt = s.mt + (int64_t)tk.mt_slot * NB * NB;
    for (int q = tid; q < w * NB; q += 256) {
        const int i = q / NB, j = q % NB;
        if (j >= w) continue;
        double v = i <= j ? X[j * DLD + i] * p0[j] : 0.0;
        if (p1[j] != 0.0) {
            const int o = de[j] != 0.0 ? j + 1 : j - 1;
            if (i <= o) v += X[o * DLD + i] * p1[j];
        }
        mt[perm[i] * NB + j] = (T)v;
    }
    int dummy = 0;
    lmax = warp_max_key(lmax, dummy);
    if (lane == 0 && lmax) atomicMax(&s.counts[6], lmax);
    if (tid == 0) {
        atomicAdd(&s.counts[0], c_neg);
        atomicAdd(&s.counts[1], c_zero);
        atomicAdd(&s.counts[2], c_pos);
        if (c_tiny) atomicAdd(&s.counts[3], c_tiny);
        double ratio = s_minpiv / (s.norm > 0 ? s.norm : 1.0);
        atomicMin(&s.counts[4], (unsigned long long)__double_as_longlong(ratio));
        if (c_2x2) atomicAdd(&s.counts[5], c_2x2);
    }
}

// ---------------------------------------------------------------- K4: panel transform
// Block = (task, 16 RA rows of a 64-row tile).  L21 = F21 Mt written in place; W = L21 D to
// scratch.  In the pivot order Mt is L^-T D^-1, upper triangular but for the 2x2 pivots' entries
// just below its diagonal, so column quarter b takes terms 0 .. 16 (b + 1) only.  The FP64 pipe
// bounds it (43 us for 64 rows on one SM): steps with few tiles split them over more SMs (RA).
// Dynamic shared memory: panel_smem<T, RA>().
template <typename T, int RA>
__global__ void __launch_bounds__(256) k_panel(const StepTask *__restrict__ tasks, int32_t ntask,
                                                const ShiftPtrs<T> *sp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int RT = 16 * RA, LDR = RT + 1, SUB = TR / RT;
    T (*Ms)[NB + 1] = reinterpret_cast<T (*)[NB + 1]>(smem_raw);                       // Ms[t][j]
    T (*Fs)[LDR] = reinterpret_cast<T (*)[LDR]>(smem_raw + sizeof(T) * NB * (NB + 1));   // Fs[t][row]
    T (*Ls)[LDR] = reinterpret_cast<T (*)[LDR]>(smem_raw + sizeof(T) * NB * (NB + 1 + LDR));
    __shared__ double sd[NB], se[NB];
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const int32_t tile = blockIdx.x / SUB;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].tiles4_pre <= tile) lo = mid; else hi = mid - 1;
    }
    const StepTask tk = tasks[lo];
    const int w = tk.w, m = tk.m;
    const int r0 = (tile - tk.tiles4_pre) * TR + (int)(blockIdx.x % SUB) * RT;   // first row within the r rows
    const int nr = min(RT, tk.r - r0);
    if (nr <= 0) return;
    T *F = s.ws + tk.front_off;
    const int64_t rowbase = tk.k0 + w + r0;
    const T *mt = s.mt + (int64_t)tk.mt_slot * NB * NB;
    const int32_t *pv = s.piv + (int64_t)tk.panel * NB;
    const int tid = threadIdx.x;
    for (int q = tid; q < NB * RT; q += 256) {
        const int t = q / RT, i = q % RT;
        Fs[t][i] = (t < w && i < nr) ? F[(int64_t)(tk.k0 + pv[t]) * m + rowbase + i] : (T)0;
    }
    for (int q = tid; q < NB * NB; q += 256) {
        const int t = q / NB, j = q % NB;
        Ms[t][j] = (t < w && j < w) ? mt[pv[t] * NB + j] : (T)0;
    }
    if (tid < NB) {
        sd[tid] = tid < w ? s.dblk[(int64_t)tk.panel * 2 * NB + tid] : 0.0;
        se[tid] = tid < w ? s.dblk[(int64_t)tk.panel * 2 * NB + NB + tid] : 0.0;
    }
    __syncthreads();
    // each thread: rows i = tx + 16 a, cols j = ty + 16 b
    const int tx = tid & 15, ty = tid >> 4;
    T acc[RA][4];
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        if (16 * h >= w) break;
        for (int t = 16 * h; t < min(16 * h + 16, w); ++t) {
            T fa[RA];
#pragma unroll
            for (int a = 0; a < RA; ++a) fa[a] = Fs[t][tx + 16 * a];
#pragma unroll
            for (int b = h; b < 4; ++b) {
                const T mb = Ms[t][ty + 16 * b];
#pragma unroll
                for (int a = 0; a < RA; ++a) acc[a][b] += fa[a] * mb;
            }
        }
        if (h > 0) {                                 // a 2x2 pivot across columns 16 h - 1, 16 h
            const T mb = Ms[16 * h][ty + 16 * (h - 1)];
#pragma unroll
            for (int a = 0; a < RA; ++a) acc[a][h - 1] += Fs[16 * h][tx + 16 * a] * mb;
        }
    }
#pragma unroll
    for (int a = 0; a < RA; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) Ls[ty + 16 * b][tx + 16 * a] = acc[a][b];
    __syncthreads();
    T *W = s.wbuf + tk.wbuf_off;
    unsigned long long lmax = 0;
    for (int q = tid; q < w * RT; q += 256) {
        int j = q / RT, i = q % RT;
        if (i >= nr) continue;
        T l = Ls[j][i];
        lmax = max(lmax, abs_bits((double)l));
        F[(int64_t)(tk.k0 + j) * m + rowbase + i] = l;
        double wv = (double)l * sd[j];
        if (se[j] != 0.0) wv += (double)Ls[j + 1][i] * se[j];
        if (j > 0 && se[j - 1] != 0.0) wv += (double)Ls[j - 1][i] * se[j - 1];
        W[(int64_t)j * tk.r + r0 + i] = (T)wv;
    }
    int dummy = 0;
    lmax = warp_max_key(lmax, dummy);
    if ((tid & 31) == 0 && lmax) atomicMax(&s.counts[6], lmax);
}

// ---------------------------------------------------------------- K3: Schur update
// Block = (task, lower-triangular tile pair).  C[i][j] -= sum_t L21[i][t] W[j][t].
// Dynamic shared memory: 2 * NB * (TR + 1) * sizeof(T).
template <typename T>
__global__ void __launch_bounds__(256) k_schur(const StepTask *__restrict__ tasks, int32_t ntask,
                                                const ShiftPtrs<T> *sp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T (*As)[TR + 1] = reinterpret_cast<T (*)[TR + 1]>(smem_raw);                // As[t][i] = L21[i][t]
    T (*Bs)[TR + 1] = reinterpret_cast<T (*)[TR + 1]>(smem_raw + sizeof(T) * NB * (TR + 1));
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const int32_t tile = blockIdx.x;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].tiles3_pre <= tile) lo = mid; else hi = mid - 1;
    }
    const StepTask tk = tasks[lo];
    const int q = tile - tk.tiles3_pre;
    int bi = (int)((sqrt(8.0 * q + 1.0) - 1.0) * 0.5);
    while ((bi + 1) * (bi + 2) / 2 <= q) ++bi;
    while (bi * (bi + 1) / 2 > q) --bi;
    const int bj = q - bi * (bi + 1) / 2;
    const int w = tk.w, m = tk.m, r = tk.r;
    const int i0 = bi * TR, j0 = bj * TR;
    const int ni = min(TR, r - i0), nj = min(TR, r - j0);
    T *F = s.ws + tk.front_off;
    const T *W = s.wbuf + tk.wbuf_off;
    const int64_t base = tk.k0 + w;               // first trailing row/col in the front
    const int tid = threadIdx.x;
    for (int e = tid; e < w * TR; e += 256) {
        int t = e / TR, i = e % TR;
        As[t][i] = i < ni ? F[(int64_t)(tk.k0 + t) * m + base + i0 + i] : (T)0;
        Bs[t][i] = i < nj ? W[(int64_t)t * r + j0 + i] : (T)0;
    }
    __syncthreads();
    const int tx = tid & 15, ty = tid >> 4;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
    for (int t = 0; t < w; ++t) {
        T fa[4], fb[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) fa[a] = As[t][tx + 16 * a];
#pragma unroll
        for (int b = 0; b < 4; ++b) fb[b] = Bs[t][ty + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] += fa[a] * fb[b];
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        int j = ty + 16 * b;
        if (j >= nj) continue;
        T *col = F + (base + j0 + j) * (int64_t)m + base + i0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            int i = tx + 16 * a;
            if (i < ni && i0 + i >= j0 + j) col[i] -= acc[a][b];
        }
    }
}

}  // namespace ssk
