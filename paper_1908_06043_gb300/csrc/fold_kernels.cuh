// FP64 triangular solves with the folded factor (Alg. 2 step 3: V <- L^-T D^-1 L^-1 (B V)).
//
// For a panel with pivot order P, unit lower L11 and block-diagonal D the factorisation's
// L21 is replaced, once, by G = L21 L11^-1 P (k_fold_panels).  With it a solve reads
//   forward:  b2 -= G b1                                   (every level, pushed with atomics)
//   middle:   x1 = P^T L11^-T D^-1 L11^-1 P b1             (all panels at once)
//   backward: x1 -= G^T x2                                 (every level, atomics)
// in place on the N x k right-hand sides (row-major, permuted order).  The diagonal blocks
// leave the chain of levels, so a level costs one grid barrier a sweep instead of two, and no
// panel-sized triangular product stands between two barriers.  |G| grows like |L21| times the
// inverse of a 64 x 64 unit lower triangle whose entries Bunch-Kaufman pivoting bounds; the
// error of an FP64 solve is the factor's own in both forms.  The half solve x = P L^-T y needs
// only L^-T: x1 = P^T L11^-T y1 - G^T x2.
//
// What bounds it.  FP64 runs at 2 multiply-adds a clock and SM here, and a warp issues one FP64
// instruction per 64 clocks at most: an item of 16 x 7 multiply-adds on one warp takes 7,200 clocks
// however idle the rest of the chip is.  An item is one warp's 32 rows x 16 panel columns (forward) or
// 128 rows x 4 panel columns (backward) times at most 8 right-hand sides;
// a level with few of them halves its items (columns, rows) up to three times, to eight warps an
// SM (four: 2% slower, sixteen: 3%).  Few right-hand sides are bound by the chain of levels:
// some 850 clocks for b1 (x2) from the L2, the multiply-adds, 800 until the additions are performed,
// 650 a poll of the barrier.  The entries of a warp's first item in the next level never change: they
// are fetched while the other blocks arrive, from records read one and two levels before.  The
// forward additions to a row's right-hand sides come from consecutive lanes: as one 8-byte
// reduction a lane and row they were the limit of wide levels (about 25 a clock over the chip).
// Measured (GB300, ms a solve).  Two barriers a level and sweep, a 64-row tile and its 64 x 64
// diagonal products per block / folded, whole items / now: N = 864, k = 1 1.34 / 0.09 / 0.064;
// N = 2,688, k = 4 3.6 / 0.32 / 0.20; N = 9,180, k = 7 8.7 / 1.28 / 0.89; N = 16,384, k = 1
// 17.6 / 1.2 / 0.85.  At the FP64 pipe's limit (N = 5,280, k = 304, no tensor cores) 11.7 / 10.6.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "factor_kernels.cuh"
#include "grid_sync.cuh"
#include "internal.h"

namespace ssk {

constexpr int kFoldThreads = 512;
constexpr int kFoldWarps = kFoldThreads / 32;
constexpr int kFoldRows = 128;       // rows of a tile: 16 items of either kind
constexpr int kFoldMaxNc = 8;        // right-hand sides of an item
constexpr int kMidCols = 8;          // right-hand sides of a middle item
constexpr size_t kFoldPanelsSmem = sizeof(double) * 2 * NB * (NB + 1);
// middle item: L11^-1 and the right-hand sides; level items: 128 x 8 values a warp
constexpr size_t kFoldMidSmem = sizeof(double) * (NB * (NB + 1) + NB * (kMidCols + 1) + 5 * NB);
// values a warp stages for items of nc right-hand sides: 128 rows, an odd number of values apart
__host__ __device__ constexpr int fold_ws(int nc) { return kFoldRows * (nc | 1); }
__host__ __device__ constexpr size_t fold_item_smem(int nc) { return sizeof(double) * kFoldWarps * fold_ws(nc); }
constexpr size_t kFoldItemSmem = fold_item_smem(kFoldMaxNc);
constexpr size_t kFoldUseSmem = kFoldMidSmem > kFoldItemSmem ? kFoldMidSmem : kFoldItemSmem;
// more than half an SM's shared memory: one block per SM, so that consecutive blocks -- and
// with them the items of a small level -- lie on different SMs
constexpr size_t kFoldSmem = kFoldUseSmem > 118 * 1024 ? kFoldUseSmem : 118 * 1024;

// G = L21 L11^-1 P in place in the L storage: block = (panel, 64-row tile).  P sends entry
// piv[s] of a panel to position s, so column s of L21 L11^-1 goes to column piv[s] of G.
__global__ void __launch_bounds__(256) k_fold_panels(const PanelDesc *__restrict__ panels,
                                                     const double *__restrict__ linv,
                                                     const int32_t *__restrict__ piv, double *arena) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double (*Ls)[TR + 1] = reinterpret_cast<double (*)[TR + 1]>(smem_raw);                             // [i][row]
    double (*Ms)[NB + 1] = reinterpret_cast<double (*)[NB + 1]>(smem_raw + sizeof(double) * NB * (TR + 1));   // [i][s]
    const int p = blockIdx.x;
    const PanelDesc pd = panels[p];
    const int w = pd.w, m = pd.m, r = m - pd.k0 - w, r0 = blockIdx.y * TR;
    if (r0 >= r) return;
    const int nr = min(TR, r - r0), tid = threadIdx.x;
    double *F = arena + pd.front_off;
    const int64_t rowbase = pd.k0 + w + r0;
    for (int q = tid; q < NB * TR; q += 256) {
        const int t = q / TR, i = q % TR;
        Ls[t][i] = (t < w && i < nr) ? F[(int64_t)(pd.k0 + t) * m + rowbase + i] : 0.0;
        Ms[t][i] = linv[(int64_t)p * NB * NB + q];          // zero outside the w x w triangle
    }
    __syncthreads();
    // rows tx + 16 a, columns ty + 16 b; L11^-1 is lower triangular, so terms i of the quarter
    // [16 h, 16 h + 16) reach the columns of quarters b <= h only
    const int tx = tid & 15, ty = tid >> 4;
    double acc[4][4] = {};
#pragma unroll
    for (int h = 0; h < 4; ++h)
        for (int i = 16 * h; i < min(16 * h + 16, w); ++i) {
            double l[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) l[a] = Ls[i][tx + 16 * a];
#pragma unroll
            for (int b = 0; b <= h; ++b) {
                const double mv = Ms[i][ty + 16 * b];
#pragma unroll
                for (int a = 0; a < 4; ++a) acc[a][b] += l[a] * mv;
            }
        }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int s = ty + 16 * b;
        if (s >= w) continue;
        double *col = F + (int64_t)(pd.k0 + piv[(int64_t)p * NB + s]) * m + rowbase;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (tx + 16 * a < nr) col[tx + 16 * a] = acc[a][b];
    }
}

// A tile of a panel's rows below its diagonal block, so that a block needs one load to find its
// work: entry (i, t) of G is arena[off + t m + i], its global row idx[idx + i], its global column
// g0 + t; nr rows, w columns.
struct FoldTile {
    int64_t off, idx;
    int32_t m, w, nr, g0;
};
struct FoldLevel {          // a solve level's tiles
    int32_t tile0, tiles;   // 128-row tiles (fold_kernels.cuh)
    int32_t tile0_64, tiles_64;   // 64-row tiles (fold_tc.cuh)
};

struct FoldArgs {
    const FoldLevel *lev;
    int32_t nlev, npan;
    int32_t k;
    int32_t full;           // 1: forward, D^-1 and backward; 0: L^-T only
    const FoldTile *tiles, *tiles_64;
    const PanelDesc *panels;
    const int32_t *idx;
    const double *linv;
    const double *dblk;
    const int32_t *piv;
    const double *arena;
    const int32_t *sc;      // scale exponent of every (permuted) column (fold_tc.cuh)
    GridBar *bar;
    long long limit;
};

// sc[i] = exponent of about sqrt(|a_rr| + |sigma b_rr|), r = perm[i] (i without perm); 0 where that is
// zero or not finite.  Scaling row and column i of the pencil by 2^s adds s.  Thread = row.
__global__ void k_fold_scales(int64_t n, const int32_t *__restrict__ perm, const int64_t *__restrict__ rowptr,
                              const int32_t *__restrict__ colind, const double *__restrict__ a,
                              const double *__restrict__ b, double sigma, int32_t *__restrict__ sc) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t r = perm ? perm[i] : (int32_t)i;
    int64_t lo = rowptr[r], hi = rowptr[r + 1] - 1;        // the diagonal is stored, columns ascend
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (colind[mid] < r) lo = mid + 1; else hi = mid;
    }
    const double d = fabs(a[lo]) + fabs(sigma * b[lo]);
    sc[i] = d > 0.0 && isfinite(d) ? (ilogb(d) + 1) >> 1 : 0;
}

// A level's items are halved `split` times over, until there is one for each of `slots` warps.
__host__ __device__ __forceinline__ int fold_split(int64_t items, int64_t slots) {
    int s = 0;
    while (s < 3 && (items << (s + 1)) <= slots) ++s;
    return s;
}

// The entries of G that a lane holds for one item, with where they belong.
struct FoldItem {
    double g[16];
    int32_t row[4];         // global rows of the item: forward row[0] (lane), backward lane + 32 j
    int32_t g0;             // global index of the item's first panel column
    int32_t nt;             // panel columns of the item (forward up to 16, backward up to 4); 0: empty
    int32_t nr;             // rows of the item
};

// forward item e of tile tl's level: 32 rows (one a lane), 16 >> split columns
__device__ __forceinline__ void fold_load_fwd(const FoldArgs &a, const FoldTile &tl, int split, int e, FoldItem &it) {
    const int sub = e & ((16 << split) - 1), nc = 16 >> split, lane = threadIdx.x & 31;
    const int t0 = nc * (sub & ((4 << split) - 1)), i0 = 32 * (sub >> (2 + split));
    it.nr = min(32, tl.nr - i0);
    it.nt = it.nr > 0 ? min(nc, tl.w - t0) : 0;
    it.g0 = tl.g0 + t0;
    if (it.nt <= 0) return;
    const bool in = lane < it.nr;
    it.row[0] = in ? a.idx[tl.idx + i0 + lane] : 0;
    const double *F = a.arena + tl.off + (int64_t)t0 * tl.m + i0 + lane;
#pragma unroll
    for (int u = 0; u < 16; ++u) it.g[u] = (in && u < it.nt) ? __ldg(F + (int64_t)u * tl.m) : 0.0;
}

// backward item e of tile tl's level: 128 >> split rows (lane % 8 + 8 j), 4 columns (one to 8 lanes)
__device__ __forceinline__ void fold_load_bwd(const FoldArgs &a, const FoldTile &tl, int split, int e, FoldItem &it) {
    const int sub = e & ((16 << split) - 1), nrow = kFoldRows >> split, lane = threadIdx.x & 31;
    const int t0 = 4 * (sub & 15), i0 = nrow * (sub >> 4), rg = lane & 7, t = lane >> 3;
    it.nr = min(nrow, tl.nr - i0);
    it.nt = it.nr > 0 ? min(4, tl.w - t0) : 0;
    it.g0 = tl.g0 + t0;
    if (it.nt <= 0) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) it.row[j] = lane + 32 * j < it.nr ? a.idx[tl.idx + i0 + lane + 32 * j] : 0;
    const double *F = a.arena + tl.off + (int64_t)(t0 + t) * tl.m + i0 + rg;
#pragma unroll
    for (int j = 0; j < 16; ++j) it.g[j] = (t < it.nt && rg + 8 * j < it.nr) ? __ldg(F + 8 * j) : 0.0;
}

// b2 -= G b1 for the item's rows and columns, right-hand sides [c0, c0 + NC) of k
template <int NC>
__device__ __forceinline__ void fold_fwd(const FoldItem &it, double *ws, double *b, int k, int c0) {
    if (it.nt <= 0) return;
    const int lane = threadIdx.x & 31, kc = min(NC, k - c0);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 16 * NC; e += 32) {
        const int q = e + lane, t = q / NC, c = q % NC;
        if (q < 16 * NC) ws[q] = (t < it.nt && c < kc) ? __ldcg(&b[(int64_t)(it.g0 + t) * k + c0 + c]) : 0.0;
    }
    __syncwarp();
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
#pragma unroll
    for (int u = 0; u < 16; u += 2) {
        if (u >= it.nt) break;
#pragma unroll
        for (int v = u; v < u + 2; ++v)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] += it.g[v] * ws[v * NC + c];
    }
    if constexpr (NC == 1) {
        if (lane < it.nr) atomicAdd(b + (int64_t)it.row[0] * k + c0, -acc[0]);
    } else {
        // a row's right-hand sides lie together: added by consecutive lanes they are one or two
        // sectors of the L2 a row, not NC
        constexpr int P = NC | 1;
        __syncwarp();
#pragma unroll
        for (int c = 0; c < NC; ++c) ws[lane * P + c] = -acc[c];
        __syncwarp();
#pragma unroll
        for (int u = 0; u < NC; ++u) {
            const int q = 32 * u + lane, i = q / NC, c = q % NC;
            const int row = __shfl_sync(0xffffffffu, it.row[0], i);
            if (i < it.nr && c < kc) atomicAdd(b + (int64_t)row * k + c0 + c, ws[i * P + c]);
        }
    }
}

// Sum of V values (a power of two) over the lanes that differ in the bits OFF, OFF / 2, .. 1: while
// V > 1 a lane keeps one half and passes the other on (V / 2 additions); afterwards v[0 .. *left) are
// the values base .. base + *left.
template <int V, int OFF>
__device__ __forceinline__ void fold_reduce(double *v, int lane, int &base, int &left) {
    if constexpr (OFF == 0) {
        left = V;
    } else if constexpr (V > 1) {
        const bool up = (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            const double keep = up ? v[i + V / 2] : v[i], send = up ? v[i] : v[i + V / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
        }
        base += up ? V / 2 : 0;
        fold_reduce<V / 2, OFF / 2>(v, lane, base, left);
    } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], OFF);
        fold_reduce<1, OFF / 2>(v, lane, base, left);
    }
}
// the lanes that hold a result of fold_reduce<V, OFF> alone (the others hold copies)
template <int V, int OFF>
__device__ __forceinline__ bool fold_owner(int lane) {
    if constexpr (OFF == 0) return true;
    else if constexpr (V > 1) return fold_owner<V / 2, OFF / 2>(lane);
    else return (lane & OFF) == 0 && fold_owner<1, OFF / 2>(lane);
}

// x1 -= G^T x2 for the item's rows and columns: a lane sums one column over every eighth row, so
// that NC values over 8 lanes are left to add
template <int NC>
__device__ __forceinline__ void fold_bwd(const FoldItem &it, double *ws, double *b, int k, int c0) {
    if (it.nt <= 0) return;
    constexpr int P = NC | 1;                             // distance of two rows in ws
    constexpr int V = NC <= 1 ? 1 : NC <= 2 ? 2 : NC <= 4 ? 4 : 8;
    const int lane = threadIdx.x & 31, kc = min(NC, k - c0), rg = lane & 7, t = lane >> 3;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (32 * j >= it.nr) break;
        const bool in = lane + 32 * j < it.nr;
        const double *src = b + (int64_t)it.row[j] * k + c0;
#pragma unroll
        for (int c = 0; c < NC; ++c) ws[(lane + 32 * j) * P + c] = (in && c < kc) ? __ldcg(src + c) : 0.0;
    }
    __syncwarp();
    double acc[V];
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] = 0.0;
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
        if (8 * j >= it.nr) break;
#pragma unroll
        for (int v = j; v < j + 2; ++v)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[c] += it.g[v] * ws[(rg + 8 * v) * P + c];
    }
    int base = 0, left = 0;
    fold_reduce<V, 4>(acc, lane, base, left);
    if (t >= it.nt || !fold_owner<V, 4>(lane)) return;
    double *o = b + (int64_t)(it.g0 + t) * k + c0;
#pragma unroll
    for (int e = 0; e < V; ++e) {
        if (e >= left) break;
        if (base + e < kc) atomicAdd(o + base + e, -acc[e]);
    }
}

// Middle step of a panel, right-hand sides [8 chunk, 8 chunk + 8): x1 = P^T L11^-T D^-1 L11^-1 P b1
// (full), or P^T L11^-T b1.  One block.  What does not depend on the right-hand sides comes first, so
// that the sweep kernel has it done while it waits for the forward sweep's last level: L11^-1, P, D's
// pivots (diagonal or 2 x 2 determinants) and their reciprocals -- a division is some 40 FP64
// instructions, so it is done once a row and not once a value.
struct FoldMid {
    double (*Lm)[NB + 1];
    double (*Y)[kMidCols + 1];
    double *sd, *se, *det, *rdet;      // D's diagonal and sub-diagonal, pivots, reciprocals
    int32_t *pv;
    __device__ explicit FoldMid(unsigned char *smem) {
        Lm = reinterpret_cast<double (*)[NB + 1]>(smem);
        Y = reinterpret_cast<double (*)[kMidCols + 1]>(smem + sizeof(double) * NB * (NB + 1));
        sd = reinterpret_cast<double *>(smem + sizeof(double) * (NB * (NB + 1) + NB * (kMidCols + 1)));
        se = sd + NB, det = se + NB, rdet = det + NB;
        pv = reinterpret_cast<int32_t *>(rdet + NB);
    }
};

__device__ __forceinline__ void fold_mid_load(unsigned char *smem_raw, const FoldArgs &a, int p) {
    const FoldMid m(smem_raw);
    const int tid = threadIdx.x;
    constexpr int MU = NB * NB / kFoldThreads;
    double mv[MU];
#pragma unroll
    for (int u = 0; u < MU; ++u) mv[u] = __ldg(&a.linv[(int64_t)p * NB * NB + tid + kFoldThreads * u]);
    if (tid < NB) {
        const double *D = a.dblk + (int64_t)p * 2 * NB, *E = D + NB;
        const double d = D[tid], e = E[tid], e0 = tid > 0 ? E[tid - 1] : 0.0;
        const double d0 = tid > 0 ? D[tid - 1] : 0.0, d1 = tid + 1 < NB ? D[tid + 1] : 0.0;
        const double det = e != 0.0 ? d * d1 - e * e : e0 != 0.0 ? d0 * d - e0 * e0 : d;
        m.pv[tid] = a.piv[(int64_t)p * NB + tid];
        m.sd[tid] = d;
        m.se[tid] = e;
        m.det[tid] = det;
        // beyond 2^+-1000 the reciprocal has too few bits: NaN sends the row to the division
        m.rdet[tid] = fabs(det) > 0x1p-1000 && fabs(det) < 0x1p1000 ? 1.0 / det : nan("");
    }
#pragma unroll
    for (int u = 0; u < MU; ++u) m.Lm[(tid + kFoldThreads * u) / NB][(tid + kFoldThreads * u) % NB] = mv[u];
}

// after fold_mid_load and a __syncthreads().  Thread = (row i, column c, part ts of the dot product):
// MC columns and 8 / MC parts share a row's 8 lanes, so few right-hand sides still fill the lanes.
template <int MC>
__device__ __forceinline__ void fold_mid(unsigned char *smem_raw, const FoldArgs &a, int p, int chunk, double *b) {
    const FoldMid m(smem_raw);
    constexpr int TS = 8 / MC;
    const int w = a.panels[p].w, g0 = a.panels[p].g0;
    const int tid = threadIdx.x, i = tid >> 3, c = tid & (MC - 1), ts = (tid & 7) / MC;
    const int k = a.k, c0 = chunk * MC;
    const bool in = i < w && c0 + c < k;
    const int pv = i < w ? m.pv[i] : 0;
    if (ts == 0) m.Y[i][c] = in ? __ldcg(&b[(int64_t)(g0 + (a.full ? pv : i)) * k + c0 + c]) : 0.0;
    __syncthreads();
    double s = 0.0, s1 = 0.0;
    if (a.full) {
        for (int t = ts; t <= i; t += 2 * TS) {           // Lm is zero above its diagonal
            s += m.Lm[i][t] * m.Y[t][c];
            if (t + TS < NB) s1 += m.Lm[i][t + TS] * m.Y[t + TS][c];
        }
        s += s1;
#pragma unroll
        for (int o = MC; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __syncthreads();
        if (ts == 0) m.Y[i][c] = i < w ? s : 0.0;
        __syncthreads();
        const int r = tid / MC, q = tid % MC;             // in as few warps as the values fill
        double u = 0.0;
        if (r < w && c0 + q < k) {
            // rows of a 2 x 2 block [A B; B C]: (C y0 - B y1) / det and (A y1 - B y0) / det
            const bool first = m.se[r] != 0.0, second = r > 0 && m.se[r - 1] != 0.0;
            const int o = first ? r + 1 : second ? r - 1 : r;
            const double f = first ? -m.se[r] : second ? -m.se[r - 1] : 0.0;
            const double num = first || second ? f * m.Y[o][q] + m.sd[o] * m.Y[r][q] : m.Y[r][q];
            const double det = m.det[r], rd = m.rdet[r];
            u = num * rd;
            u += rd * fma(-u, det, num);                  // the quotient, to about its last bit
            if (!isfinite(u)) u = det != 0.0 || first || second ? num / det : 0.0;
        }
        __syncthreads();
        if (r < NB) m.Y[r][q] = u;
        __syncthreads();
    }
    s = 0.0, s1 = 0.0;
    for (int t = (i / (2 * TS)) * (2 * TS) + ts; t < w; t += 2 * TS) {
        s += m.Lm[t][i] * m.Y[t][c];
        if (t + TS < NB) s1 += m.Lm[t + TS][i] * m.Y[t + TS][c];
    }
    s += s1;
#pragma unroll
    for (int o = MC; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (in && ts == 0) b[(int64_t)(g0 + pv) * k + c0 + c] = s;
}

__device__ __forceinline__ void fold_mid_any(unsigned char *smem_raw, const FoldArgs &a, int mc, int p, int chunk, double *b) {
    if (mc == 1) fold_mid<1>(smem_raw, a, p, chunk, b);
    else if (mc == 2) fold_mid<2>(smem_raw, a, p, chunk, b);
    else if (mc == 4) fold_mid<4>(smem_raw, a, p, chunk, b);
    else fold_mid<8>(smem_raw, a, p, chunk, b);
}
// columns a middle item takes: as many as k fills, unless fewer leave less of nb blocks' last
// round of items empty (an item costs its columns and, for L11^-1, about one more)
__host__ __device__ __forceinline__ int fold_mid_cols(int k, int npan, int nb) {
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int mc = k == 1 ? 1 : k == 2 ? 2 : k <= 4 ? 4 : 8; mc >= 1; mc >>= 1) {
        const int64_t items = (int64_t)npan * ((k + mc - 1) / mc), c = (items + nb - 1) / nb * (mc + 1);
        if (c < cost) { cost = c; best = mc; }
    }
    return best;
}

// Both sweeps in one cooperative launch: level by level, a bounded grid barrier between levels.
// Item q of a level goes to warp q / gridDim.x of block q % gridDim.x.  On a barrier timeout
// bar->err is set and every block returns.
template <int NC>
__global__ void __launch_bounds__(kFoldThreads, 1) k_fold_sweeps(const FoldArgs a, double *b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int k = a.k, nch = (k + NC - 1) / NC;
    const int nb = gridDim.x, q0 = (threadIdx.x >> 5) * nb + blockIdx.x, nw = kFoldWarps * nb;
    double *ws = reinterpret_cast<double *>(smem_raw) + (threadIdx.x >> 5) * fold_ws(NC);
    // A level's record is read two levels ahead and this warp's first tile one ahead, so that after a
    // level's work only the entries of the next one's first item are left to fetch, while the other
    // blocks arrive.
    struct Level {
        FoldLevel lv;
        int split, per;                     // items of a chunk of right-hand sides
    } cur, nxt;
    auto shape = [&](const FoldLevel &lv) {
        const int s = fold_split((int64_t)lv.tiles * 16 * nch, kFoldWarps / 2 * nb);
        return Level{lv, s, lv.tiles * (16 << s)};
    };
    auto item = [&](const Level &l, int q) { return nch == 1 ? q : q % l.per; };
    auto tile = [&](const Level &l, int q) { return a.tiles[l.lv.tile0 + (item(l, q) >> (4 + l.split))]; };
    const int mc = fold_mid_cols(k, a.npan, nb), nmid = a.npan * ((k + mc - 1) / mc);
    FoldItem it;
    FoldTile tn{};
    FoldLevel after{};
    unsigned int at = 0;
    if (a.full) {
        cur = shape(a.lev[0]);
        if (q0 < cur.per * nch) fold_load_fwd(a, tile(cur, q0), cur.split, item(cur, q0), it);
        if (a.nlev > 1) after = a.lev[1];
        for (int L = 0; L < a.nlev; ++L) {
            const bool more = L + 1 < a.nlev;
            nxt = shape(more ? after : FoldLevel{0, 0, 0, 0});
            const bool has = q0 < nxt.per * nch;
            if (has) tn = tile(nxt, q0);
            if (L + 2 < a.nlev) after = a.lev[L + 2];
            for (int q = q0; q < cur.per * nch; q += nw) {
                if (q != q0) fold_load_fwd(a, tile(cur, q), cur.split, item(cur, q), it);
                fold_fwd<NC>(it, ws, b, k, nch == 1 ? 0 : (q / cur.per) * NC);
            }
            const bool any = cur.lv.tiles > 0;
            const bool last = !more || (L + 2 == a.nlev && nxt.per == 0);      // the root has no rows below
            if (any) grid_arrive(a.bar, nb, at);
            if (has) fold_load_fwd(a, tn, nxt.split, item(nxt, q0), it);
            if (last && blockIdx.x < nmid) fold_mid_load(smem_raw, a, blockIdx.x % a.npan);
            if (any && !grid_wait(a.bar, a.limit, at)) return;
            if (last) break;
            cur = nxt;
        }
    }
    for (int q = blockIdx.x; q < nmid; q += nb) {
        __syncthreads();
        if (q != blockIdx.x || !a.full) {
            fold_mid_load(smem_raw, a, q % a.npan);
            __syncthreads();
        }
        fold_mid_any(smem_raw, a, mc, q % a.npan, q / a.npan, b);
    }
    grid_arrive(a.bar, nb, at);
    cur = shape(a.lev[a.nlev - 1]);
    if (q0 < cur.per * nch) fold_load_bwd(a, tile(cur, q0), cur.split, item(cur, q0), it);
    if (a.nlev > 1) after = a.lev[a.nlev - 2];
    if (!grid_wait(a.bar, a.limit, at)) return;
    for (int L = a.nlev - 1; L >= 0; --L) {
        nxt = shape(L > 0 ? after : FoldLevel{0, 0, 0, 0});
        const bool has = q0 < nxt.per * nch;
        if (has) tn = tile(nxt, q0);
        if (L > 1) after = a.lev[L - 2];
        for (int q = q0; q < cur.per * nch; q += nw) {
            if (q != q0) fold_load_bwd(a, tile(cur, q), cur.split, item(cur, q), it);
            fold_bwd<NC>(it, ws, b, k, nch == 1 ? 0 : (q / cur.per) * NC);
        }
        if (L == 0) break;
        const bool any = cur.lv.tiles > 0;
        if (any) grid_arrive(a.bar, nb, at);
        if (has) fold_load_bwd(a, tn, nxt.split, item(nxt, q0), it);
        if (any && !grid_wait(a.bar, a.limit, at)) return;
        cur = nxt;
    }
}

// one level of one sweep per launch (SS_SOLVE_PER_STEP, ss_solve_noalloc): warp = item
template <int NC>
__global__ void __launch_bounds__(kFoldThreads) k_fold_level(const FoldArgs a, int level, int split, int backward, double *b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *ws = reinterpret_cast<double *>(smem_raw) + (threadIdx.x >> 5) * fold_ws(NC);
    const int nch = (a.k + NC - 1) / NC;
    const FoldLevel lv = a.lev[level];
    const int64_t per = (int64_t)lv.tiles * (16 << split), q = (int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5);
    if (q >= per * nch) return;
    FoldItem it;
    const int c0 = (int)(q / per) * NC, e = (int)(q % per);
    const FoldTile tl = a.tiles[lv.tile0 + (e >> (4 + split))];
    if (backward) {
        fold_load_bwd(a, tl, split, e, it);
        fold_bwd<NC>(it, ws, b, a.k, c0);
    } else {
        fold_load_fwd(a, tl, split, e, it);
        fold_fwd<NC>(it, ws, b, a.k, c0);
    }
}

// middle step of every panel: block = (panel, chunk of right-hand sides)
__global__ void __launch_bounds__(kFoldThreads) k_fold_mid(const FoldArgs a, int mc, double *b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fold_mid_load(smem_raw, a, blockIdx.x);
    __syncthreads();
    fold_mid_any(smem_raw, a, mc, blockIdx.x, blockIdx.y, b);
}

}  // namespace ssk
