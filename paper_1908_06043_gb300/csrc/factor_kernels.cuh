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
// One block per (front, shift).  FP64 runs at 2 multiply-adds a clock and SM here and at one warp
// instruction per 64 clocks and warp, so the block does only the lower triangle's (w^3 / 6) and the
// inverse's (w^3 / 6), with one multiply-add each and no division in a loop; pivots are compared as
// integers (|x| orders like its bits).  The chain of columns is the limit: warp 0 runs one column
// ahead of the others.  It updates column k + 1, finds its largest entry and, where the diagonal fails
// the 1x1 test -- every other column of the shifted pencils -- row r of that entry, in registers; it
// decides on the pivot and forms that column of L while 12 other warps write the trailing triangle
// from one buffer to the other (6 are too few to cover their shared-memory loads).  A swap of k and r
// is part of that copy, so a column costs one block barrier whether it swaps or not; only 2x2 pivots
// move rows in place and take barriers of their own.  The three warps on warp 0's scheduler rest, one
// keeps the books.  A column takes 1,150 - 1,600 clocks, with a failed test 2,200 - 2,900; the inverse
// 28,000.  N = 16,384, 164 steps, us a step: 330 with the full square updated by three FP64 operations
// an entry behind a whole-block barrier per action and a serial column-per-thread inverse; 118 with
// the triangle updated in place, the column ahead and a failed test resolved behind three more
// barriers; 91 now.  The tests in FP32 with FP64 for near ties instead: no change.
constexpr int DLD = NB + 4;        // row stride: 8 x 4 patches touch every shared-memory bank once
constexpr int kDiagThreads = 512;
// two copies of the triangle; strict lower L, transposed, in the second one's upper half
constexpr size_t kDiagSmem = 2 * NB * DLD * sizeof(double);

__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ double from_bits(unsigned long long b) { return __longlong_as_double((long long)b); }

// largest key over the warp
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    return ((unsigned long long)mh << 32) | __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
}
// and the smallest index holding it
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long key, int &idx) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    idx = (int)__reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? (unsigned)idx : 0x7fffffffu);
    return ((unsigned long long)mh << 32) | ml;
}

// 1 / d (0 for d = 0) from the hardware's approximation x by one step of Chebyshev's third-order
// iteration (the hyperpower method of order three, Altman 1960): with e = 1 - d x,
// 1 / d = x (1 + e + e^2 + ..).  The approximation takes and gives 20 bits of mantissa, so |e| < 2^-18 and
// what is left out, e^3, is below half a unit in the last place; with the last rounding the result is
// within one unit of 1 / d (3 of 10,000 random d differ from the division).  Three dependent
// multiply-adds; a division takes some ten, and checks.  Outside 2^+-1000: the division.
__device__ __forceinline__ double diag_recip(double d) {
    const unsigned ex = (unsigned)(__double_as_longlong(d) >> 52) & 0x7ffu;
    if (ex - 23u > 2000u) return d != 0.0 ? 1.0 / d : 0.0;
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
    const double e = fma(-d, x, 1.0);
    return fma(x, fma(e, e, e), x);
}

__global__ void k_recip_selftest(int64_t n, const double *__restrict__ d, double *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = diag_recip(d[i]);
}

template <typename T>
__global__ void __launch_bounds__(kDiagThreads, 1) k_diag_bk(const StepTask *__restrict__ tasks, const ShiftPtrs<T> *sp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *buf = reinterpret_cast<double *>(smem_raw);     // lower triangle, entry (i, j) at i DLD + j
    double *L = buf + NB * DLD;                              // L(i, j), i > j, at j DLD + i
    const ShiftPtrs<T> s = sp[blockIdx.y];
    const StepTask tk = tasks[blockIdx.x];
    const int w = tk.w, m = tk.m, k0 = tk.k0;
    __shared__ int perm[NB];
    __shared__ double dd[NB], de[NB], p0[NB], p1[NB];
    __shared__ double s_y[2][NB], s_l[2][NB], s_d[2];        // the pivot's column of A and of L, the pivot
    __shared__ int s_kind[2], s_r[2];
    __shared__ unsigned long long c_neg, c_zero, c_pos, c_tiny, c_2x2, s_ratio;
    __shared__ double s_minpiv;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T *F = s.ws + tk.front_off;

    for (int q = tid; q < NB * NB; q += kDiagThreads) {
        const int j = q / NB, i = q % NB;                    // column j, row i (coalesced on i)
        if (i >= j && i < w) buf[i * DLD + j] = (double)F[(int64_t)(k0 + j) * m + (k0 + i)];
        if (i > j) L[j * DLD + i] = 0.0;
    }
    if (tid < NB) { perm[tid] = tid; dd[tid] = 0.0; de[tid] = 0.0; }
    if (tid == 0) {
        c_neg = c_zero = c_pos = c_tiny = c_2x2 = 0;
        s_minpiv = 1e300;
    }
    __syncthreads();

    const double alpha = 0.6403882032022076;   // (1 + sqrt(17)) / 8
    // Warp 0: the pivot of column c, by Bunch-Kaufman's test restricted to the block, from the
    // trailing matrix get(i, j), i >= j >= c, whose column c goes to `out`: kind 1 (1x1 at c), 2 (1x1,
    // swap c <-> r) or 3 (2x2, swap c + 1 <-> r); for 1 and 2 the column after the swap, in s_y, s_l.
    auto decide = [&](int c, int slot, double *out, auto get) {
        const int i0 = c + lane, i1 = i0 + 32;
        const bool long_col = c + 32 < w;
        double v0 = i0 < w ? get(i0, c) : 0.0, v1 = 0.0;
        if (long_col && i1 < w) v1 = get(i1, c);
        double d = __shfl_sync(0xffffffffu, v0, 0), inv = diag_recip(d);
        if (out) {
            if (i0 < w) out[i0 * DLD + c] = v0;
            if (long_col && i1 < w) out[i1 * DLD + c] = v1;
        }
        unsigned long long key = lane > 0 ? abs_bits(v0) : 0;
        int r = i0;
        if (abs_bits(v1) > key) { key = abs_bits(v1); r = i1; }
        key = warp_max_key(key, r);
        int kind = 1;
        // the test |d| < alpha lam; FP64 arithmetic only for |d| between lam / 2 and lam
        const unsigned long long kd = abs_bits(d);
        if (kd < key && key <= 0x7ff0000000000000ull) {
            const double lam = from_bits(key), akk = fabs(d);
            if (kd + (1ull << 52) <= key || akk < alpha * lam) {
                double w0 = 0.0, w1 = 0.0;
                if (i0 < w) w0 = get(max(r, i0), min(r, i0));
                if (long_col && i1 < w) w1 = get(max(r, i1), min(r, i1));
                const double h = __shfl_sync(0xffffffffu, r - c >= 32 ? w1 : w0, (r - c) & 31);
                unsigned long long ks = i0 != r ? abs_bits(w0) : 0;
                if (i1 != r && abs_bits(w1) > ks) ks = abs_bits(w1);
                const double inv_h = diag_recip(h);          // beside the tests, not after them
                const double sig = from_bits(warp_max_key(ks));
                if (!(akk * sig >= alpha * lam * lam)) {
                    kind = fabs(h) >= alpha * sig ? 2 : 3;
                    d = h;
                    inv = inv_h;
                    if (i0 != r) v0 = w0;
                    if (i1 != r) v1 = w1;
                }
            }
        }
        if (kind <= 2) {
            if (lane > 0 && i0 < w) { s_y[slot][i0] = v0; s_l[slot][i0] = v0 * inv; }
            if (long_col && i1 < w) { s_y[slot][i1] = v1; s_l[slot][i1] = v1 * inv; }
        }
        if (lane == 0) { s_kind[slot] = kind; s_r[slot] = kind == 1 ? c : r; s_d[slot] = d; }
    };
    // The trailing triangle from row / column b0, put(i, j, get(i, j)): strips of 8 rows, each cut
    // into 8 x 4 patches dealt to the warps of its strip.  A lane keeps its row in a strip, so a patch
    // is a few instructions -- with few warps a scheduler, dependent instructions, not the FP64 pipe,
    // are what an update waits for.  Warp u of n has part `part` of `parts` of strip `strip`, the
    // lowest (longest) strips have the most warps; that only changes when the first strip does.
    int strip = 0, part = 0, parts = 0;
    auto deal = [&](int b0, int u, int n) {
        const int s0 = b0 >> 3, ns = ((w + 7) >> 3) - s0, per = n / ns, more = n - per * ns;   // ns <= 8 <= n
        const bool lower = u < more * (per + 1);
        parts = lower ? per + 1 : per;
        u -= lower ? 0 : more * (per + 1);
        strip = u / parts;
        part = u - strip * parts;
        strip = s0 + ns - 1 - strip - (lower ? 0 : more);
    };
    auto patches = [&](int b0, auto get, auto put) {
        const int i = 8 * strip + (lane >> 2), step = 4 * parts;
        if (i >= w) return;
        for (int j = (b0 & ~3) + 4 * part + (lane & 3); j <= i; j += 4 * step) {
            double v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = j + q * step;
                v[q] = c >= b0 && c <= i ? get(i, c) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = j + q * step;
                if (c >= b0 && c <= i) put(i, c, v[q]);
            }
        }
    };
    int half = 0, slot = 0, first = -1;          // first strip of deal()
    if (warp == 0) decide(0, 0, nullptr, [&](int i, int j) { return buf[i * DLD + j]; });
    __syncthreads();
    for (int k = 0; k < w; slot ^= 1) {
        const int kind = s_kind[slot], r = s_r[slot];
        double *A = buf + half * NB * DLD;
        if (kind <= 2) {
            double *B = buf + (half ^ 1) * NB * DLD;
            const double *y = s_y[slot], *l = s_l[slot];
            // entry (i, j), k < j <= i, after the swap k <-> r and the pivot
            auto get = [&](int i, int j) {
                const int q = i == r ? (j == r ? k * DLD + k : j * DLD + k) : (j == r ? i * DLD + k : i * DLD + j);
                return A[q] - l[i] * y[j];
            };
            auto get1 = [&](int i, int j) { return A[i * DLD + j] - l[i] * y[j]; };      // without a swap
            if (warp == 0) {
                if (k + 1 >= w) {
                } else if (kind == 1) decide(k + 1, slot ^ 1, B, get1);
                else decide(k + 1, slot ^ 1, B, get);
            } else if (warp == 4) {
                for (int i = k + 1 + lane; i < w; i += 32) L[k * DLD + i] = l[i];
                if (kind == 2)
                    for (int j = lane; j < k; j += 32) {
                        const double t = L[j * DLD + k];
                        L[j * DLD + k] = L[j * DLD + r];
                        L[j * DLD + r] = t;
                    }
                if (lane == 0) {
                    if (kind == 2) { const int t = perm[k]; perm[k] = perm[r]; perm[r] = t; }
                    const double d = s_d[slot];
                    const unsigned long long ad = abs_bits(d), inf = 0x7ff0000000000000ull;
                    dd[k] = d;
                    if (ad == 0 || ad > inf) c_zero++; else if (__double_as_longlong(d) < 0) c_neg++; else c_pos++;
                    if (ad < abs_bits(s.tiny_thr)) c_tiny++;
                    if (ad < abs_bits(s_minpiv)) s_minpiv = from_bits(ad);
                }
                __syncwarp();
            } else if ((warp & 3) && k + 2 < w) {
                if (first != (k + 2) >> 3) {
                    first = (k + 2) >> 3;
                    deal(k + 2, 3 * (warp >> 2) + (warp & 3) - 1, 3 * kDiagThreads / 128);
                }
                auto put = [&](int i, int j, double v) { B[i * DLD + j] = v; };
                if (kind == 1) patches(k + 2, get1, put);
                else patches(k + 2, get, put);
            }
            __syncthreads();
            half ^= 1;
            k += 1;
        } else {
            const int a1 = k + 1;
            if (a1 != r) {                               // symmetric swap a1 <-> r of A, row swap of L
                if (tid < w && tid != r) {
                    const int j = tid;
                    double *x, *y;
                    if (j < k) { x = &L[j * DLD + a1]; y = &L[j * DLD + r]; }
                    else if (j < a1) { x = &A[a1 * DLD + j]; y = &A[r * DLD + j]; }
                    else if (j == a1) { x = &A[a1 * DLD + a1]; y = &A[r * DLD + r]; }
                    else if (j < r) { x = &A[j * DLD + a1]; y = &A[r * DLD + j]; }
                    else { x = &A[j * DLD + a1]; y = &A[j * DLD + r]; }
                    const double t = *x;
                    *x = *y;
                    *y = t;
                }
                if (tid == 0) { const int t = perm[a1]; perm[a1] = perm[r]; perm[r] = t; }
                __syncthreads();
            }
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
                L[k * DLD + i] = (c * ci0 - b * ci1) * id;
                L[(k + 1) * DLD + i] = (-b * ci0 + a * ci1) * id;
            }
            __syncthreads();
            if (k + 2 < w) deal(k + 2, warp, kDiagThreads / 32);
            first = -1;
            if (k + 2 < w) patches(k + 2, [&](int i, int j) {
                double v = A[i * DLD + j];
                v -= L[k * DLD + i] * A[j * DLD + k];
                v -= L[(k + 1) * DLD + i] * A[j * DLD + k + 1];
                return v;
            }, [&](int i, int j, double v) { A[i * DLD + j] = v; });
            __syncthreads();
            if (warp == 0 && k + 2 < w) decide(k + 2, slot ^ 1, nullptr, [&](int i, int j) { return A[i * DLD + j]; });
            __syncthreads();
            k += 2;
        }
    }
    // X = L^-1 in the first copy's place, by 8 x 8 diagonal blocks and three levels of
    // X21 = -X22 (L21 X11); the products L21 X11 rest in blocks above the diagonal meanwhile
    double *X = buf;
    if (tid < NB) {
        const int b = tid & ~7, jl = tid & 7;
        double x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = i == jl ? 1.0 : 0.0;
#pragma unroll
        for (int t = 0; t < 7; ++t)
#pragma unroll
            for (int i = t + 1; i < 8; ++i) x[i] -= L[(b + t) * DLD + b + i] * x[t];
#pragma unroll
        for (int i = 0; i < 8; ++i) X[(b + i) * DLD + tid] = x[i];
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
        if (tid == 2 * NB) s_ratio = (unsigned long long)__double_as_longlong(s_minpiv / (s.norm > 0 ? s.norm : 1.0));
    }
    __syncthreads();
    {
        const int C = 16 * (tid >> 6), R = C + 8, i = (tid >> 3) & 7, j = tid & 7;
        double acc = 0.0;
        if (tid < 4 * NB) {
#pragma unroll
            for (int t = 0; t < 8; ++t) acc += L[(C + t) * DLD + R + i] * X[(C + t) * DLD + C + j];
            X[(C + i) * DLD + R + j] = acc;
        }
        __syncthreads();
        if (tid < 4 * NB) {
            acc = 0.0;
#pragma unroll
            for (int t = 0; t < 8; ++t) acc += X[(R + i) * DLD + R + t] * X[(C + t) * DLD + R + j];
            X[(R + i) * DLD + C + j] = -acc;
        }
        __syncthreads();
    }
    {
        const int h = lane & 15, C = 32 * (lane >> 4), R = C + 16;
#pragma unroll
        for (int j = warp; j < 16; j += kDiagThreads / 32) {
            double acc = 0.0;
            for (int t = j; t < 16; ++t) acc += L[(C + t) * DLD + R + h] * X[(C + t) * DLD + C + j];
            X[(C + h) * DLD + R + j] = acc;
        }
        __syncthreads();
#pragma unroll
        for (int i = warp; i < 16; i += kDiagThreads / 32) {
            double acc = 0.0;
            for (int t = 0; t <= i; ++t) acc += X[(R + i) * DLD + R + t] * X[(C + t) * DLD + R + h];
            X[(R + i) * DLD + C + h] = -acc;
        }
        __syncthreads();
        if (w > 32) {
#pragma unroll
            for (int j = warp; j < 32; j += kDiagThreads / 32) {
                double acc = 0.0;
                for (int t = j; t < 32; ++t) acc += L[t * DLD + 32 + lane] * X[t * DLD + j];
                X[lane * DLD + 32 + j] = acc;
            }
            __syncthreads();
#pragma unroll
            for (int i = warp; i < 32; i += kDiagThreads / 32) {
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
    for (int q = tid; q < NB * NB; q += kDiagThreads) {
        const int i = q / NB, j = q % NB;
        linv[q] = (i < w && j <= i) ? X[i * DLD + j] : 0.0;
        if (j > i) lmax = max(lmax, abs_bits(L[i * DLD + j]));
    }
    if (tid < NB) {
        s.dblk[(int64_t)p * 2 * NB + tid] = tid < w ? dd[tid] : 0.0;
        s.dblk[(int64_t)p * 2 * NB + NB + tid] = tid < w ? de[tid] : 0.0;
        s.piv[(int64_t)p * NB + tid] = tid < w ? perm[tid] : tid;
    }
    // Mt[perm[i]][j] = sum_{t in block(j)} Li[t][i] Dinv[t][j]
    T *mt = s.mt + (int64_t)tk.mt_slot * NB * NB;
    for (int q = tid; q < w * NB; q += kDiagThreads) {
        const int i = q / NB, j = q % NB;
        if (j >= w) continue;
        double v = i <= j ? X[j * DLD + i] * p0[j] : 0.0;
        if (p1[j] != 0.0) {
            const int o = de[j] != 0.0 ? j + 1 : j - 1;
            if (i <= o) v += X[o * DLD + i] * p1[j];
        }
        mt[perm[i] * NB + j] = (T)v;
    }
    lmax = warp_max_key(lmax);
    if (lane == 0 && lmax) atomicMax(&s.counts[6], lmax);
    if (tid == 0) {
        atomicAdd(&s.counts[0], c_neg);
        atomicAdd(&s.counts[1], c_zero);
        atomicAdd(&s.counts[2], c_pos);
        if (c_tiny) atomicAdd(&s.counts[3], c_tiny);
        atomicMin(&s.counts[4], s_ratio);
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
    lmax = warp_max_key(lmax);
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
