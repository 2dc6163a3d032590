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
// What bounds it.  FP64 runs at 2 multiply-adds a clock and SM here, so the work is split until
// every SM has some: an item is one warp's 32 rows x 16 panel columns (forward) or 128 rows x 4
// panel columns (backward) times at most 8 right-hand sides, one multiply-add per entry and
// column.  Few right-hand sides are bound by the chain of levels: each warp loads the entries of
// its next level's first item (they never change) before it waits at the barrier, so a level is
// one barrier, one load of b1 (x2), a few multiply-adds and one atomic.  Measured (GB300, one
// solve; before: two barriers a level and sweep, a 64-row tile and its 64 x 64 diagonal products
// per block): N = 864, k = 1 1.34 -> 0.11 ms; N = 2,688, k = 4 3.6 -> 0.39 ms; N = 16,384, k = 1
// 17.6 -> 1.27 ms (4.9 us a level); k = 304, at the FP64 pipe's limit, 61.6 -> 61.8 ms.
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
// middle item: L11^-1 and the right-hand sides; level items: 16 x 8 values a warp
constexpr size_t kFoldMidSmem = sizeof(double) * (NB * (NB + 1) + NB * (kMidCols + 1) + 2 * NB);
constexpr size_t kFoldItemSmem = sizeof(double) * kFoldWarps * 16 * kFoldMaxNc;
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
    GridBar *bar;
    long long limit;
};

// The 16 entries of G that a lane holds for one item, with where they belong.
struct FoldItem {
    double g[16];
    int32_t row[4];         // global rows of the lane's entries (forward: row[0])
    int32_t g0;             // global index of the item's first panel column
    int32_t live;           // bit j: row[j] exists; 0 and nt = 0: an empty item
    int32_t nt;             // panel columns of the item
};

// forward item `sub` of a tile: rows 32 (sub / 4) .. + 31 (one a lane), columns 16 (sub % 4) .. + 15
__device__ __forceinline__ void fold_load_fwd(const FoldArgs &a, const FoldLevel &lv, int e, FoldItem &it) {
    const FoldTile tl = a.tiles[lv.tile0 + (e >> 4)];
    const int sub = e & 15, t0 = 16 * (sub & 3), i0 = 32 * (sub >> 2), i = i0 + (threadIdx.x & 31);
    it.nt = i0 < tl.nr ? min(16, tl.w - t0) : 0;
    it.live = i < tl.nr ? 1 : 0;
    it.g0 = tl.g0 + t0;
    if (it.nt <= 0) return;
    it.row[0] = it.live ? a.idx[tl.idx + i] : 0;
    const double *F = a.arena + tl.off + (int64_t)t0 * tl.m + i;
#pragma unroll
    for (int u = 0; u < 16; ++u) it.g[u] = (it.live && u < it.nt) ? __ldg(F + (int64_t)u * tl.m) : 0.0;
}

// backward item `sub` of a tile: its 128 rows (lane + 32 j), columns 4 sub .. + 3
__device__ __forceinline__ void fold_load_bwd(const FoldArgs &a, const FoldLevel &lv, int e, FoldItem &it) {
    const FoldTile tl = a.tiles[lv.tile0 + (e >> 4)];
    const int t0 = 4 * (e & 15);
    it.nt = min(4, tl.w - t0);
    it.live = 0;
    it.g0 = tl.g0 + t0;
    if (it.nt <= 0) return;
    const double *F = a.arena + tl.off + (int64_t)t0 * tl.m;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int i = (int)(threadIdx.x & 31) + 32 * j;
        const bool in = i < tl.nr;
        it.live |= (in ? 1 : 0) << j;
        it.row[j] = in ? a.idx[tl.idx + i] : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) it.g[4 * j + u] = (in && u < it.nt) ? __ldg(F + (int64_t)u * tl.m + i) : 0.0;
    }
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
    for (int u = 0; u < 16; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] += it.g[u] * ws[u * NC + c];
    if (!it.live) return;
    double *o = b + (int64_t)it.row[0] * k + c0;
#pragma unroll
    for (int c = 0; c < NC; ++c)
        if (c < kc) atomicAdd(o + c, -acc[c]);
}

// Sum of V values over the lanes that differ in the bits OFF, OFF / 2, .. 1: while V is even a
// lane keeps one half and passes the other on (V / 2 additions); afterwards v[0 .. *left) are the
// values base .. base + *left.
template <int V, int OFF>
__device__ __forceinline__ void fold_reduce(double *v, int lane, int &base, int &left) {
    if constexpr (OFF == 0) {
        left = V;
    } else if constexpr (V % 2 == 0) {
        const bool up = (lane & OFF) != 0;
#pragma unroll
        for (int i = 0; i < V / 2; ++i) {
            const double keep = up ? v[i + V / 2] : v[i], send = up ? v[i] : v[i + V / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, OFF);
        }
        base += up ? V / 2 : 0;
        fold_reduce<V / 2, OFF / 2>(v, lane, base, left);
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], OFF);
        fold_reduce<V, OFF / 2>(v, lane, base, left);
    }
}
// the lanes that hold a result of fold_reduce<V, 16> alone (the others hold copies)
template <int V, int OFF>
__device__ __forceinline__ bool fold_owner(int lane) {
    if constexpr (OFF == 0) return true;
    else if constexpr (V % 2 == 0) return fold_owner<V / 2, OFF / 2>(lane);
    else return (lane & OFF) == 0 && fold_owner<V, OFF / 2>(lane);
}

// x1 -= G^T x2 for the item's rows and columns
template <int NC>
__device__ __forceinline__ void fold_bwd(const FoldItem &it, double *b, int k, int c0) {
    if (it.nt <= 0) return;
    const int lane = threadIdx.x & 31, kc = min(NC, k - c0);
    double acc[4 * NC];          // [column of the panel][right-hand side]
#pragma unroll
    for (int e = 0; e < 4 * NC; ++e) acc[e] = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        double x[NC];
        const double *src = b + (int64_t)it.row[j] * k + c0;
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c] = (((it.live >> j) & 1) && c < kc) ? __ldcg(src + c) : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[u * NC + c] += it.g[4 * j + u] * x[c];
    }
    int base = 0, left = 0;
    fold_reduce<4 * NC, 16>(acc, lane, base, left);
    if (!fold_owner<4 * NC, 16>(lane)) return;
#pragma unroll
    for (int e = 0; e < 4 * NC; ++e) {
        if (e >= left) break;
        const int u = (base + e) / NC, c = (base + e) % NC;
        if (u < it.nt && c < kc) atomicAdd(&b[(int64_t)(it.g0 + u) * k + c0 + c], -acc[e]);
    }
}

// Backward items of several chunks of right-hand sides (k > kFoldMaxNc), where the FP64 pipe is
// the limit and the 31 additions a lane that fold_reduce spends on 128 multiply-adds are not:
// item `sub` of a tile is rows 16 (sub / 2) .. + 15 and columns 32 (sub % 2) .. + 31, one column a
// lane, so nothing is summed across lanes (a lane's 16 entries are one 128-byte line of its
// column).  N = 16,384, k = 304: 63.1 ms a solve with fold_bwd's items, 61.8 ms with these.
__device__ __forceinline__ void fold_load_bwd_wide(const FoldArgs &a, const FoldLevel &lv, int e, FoldItem &it) {
    const FoldTile tl = a.tiles[lv.tile0 + (e >> 4)];
    const int sub = e & 15, lane = threadIdx.x & 31, t0 = 32 * (sub & 1), i0 = 16 * (sub >> 1);
    it.nt = i0 < tl.nr ? min(32, tl.w - t0) : 0;
    it.g0 = tl.g0 + t0;
    if (it.nt <= 0) return;
    it.live = min(16, tl.nr - i0);
    it.row[0] = lane < it.live ? a.idx[tl.idx + i0 + lane] : 0;
    const double *F = a.arena + tl.off + (int64_t)(t0 + lane) * tl.m + i0;
#pragma unroll
    for (int u = 0; u < 16; ++u) it.g[u] = (u < it.live && lane < it.nt) ? __ldg(F + u) : 0.0;
}

template <int NC>
__device__ __forceinline__ void fold_bwd_wide(const FoldItem &it, double *ws, double *b, int k, int c0) {
    if (it.nt <= 0) return;
    const int lane = threadIdx.x & 31, kc = min(NC, k - c0);
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 16 * NC; e += 32) {
        const int q = e + lane, i = q / NC, c = q % NC;
        const int row = __shfl_sync(0xffffffffu, it.row[0], i & 15);
        if (q < 16 * NC) ws[q] = (i < it.live && c < kc) ? __ldcg(&b[(int64_t)row * k + c0 + c]) : 0.0;
    }
    __syncwarp();
    double acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = 0.0;
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] += it.g[u] * ws[u * NC + c];
    if (lane >= it.nt) return;
    double *o = b + (int64_t)(it.g0 + lane) * k + c0;
#pragma unroll
    for (int c = 0; c < NC; ++c)
        if (c < kc) atomicAdd(o + c, -acc[c]);
}

// Middle step of panel p, right-hand sides [8 chunk, 8 chunk + 8): x1 = P^T L11^-T D^-1 L11^-1 P b1
// (full), or P^T L11^-T b1.  One block.  Thread = (row i, column c, part ts of the dot product):
// MC columns and 8 / MC parts share a row's 8 lanes, so few right-hand sides still fill the lanes.
template <int MC>
__device__ __forceinline__ void fold_mid(unsigned char *smem_raw, const FoldArgs &a, int p, int chunk, double *b) {
    double (*Lm)[NB + 1] = reinterpret_cast<double (*)[NB + 1]>(smem_raw);
    double (*Y)[kMidCols + 1] = reinterpret_cast<double (*)[kMidCols + 1]>(smem_raw + sizeof(double) * NB * (NB + 1));
    double *sd = reinterpret_cast<double *>(smem_raw + sizeof(double) * (NB * (NB + 1) + NB * (kMidCols + 1)));
    double *se = sd + NB;
    constexpr int TS = 8 / MC;
    const PanelDesc pd = a.panels[p];
    const int tid = threadIdx.x, i = tid >> 3, c = tid & (MC - 1), ts = (tid & 7) / MC;
    const int w = pd.w, k = a.k, c0 = chunk * MC;
    const bool in = i < w && c0 + c < k;
    constexpr int MU = NB * NB / kFoldThreads;
    double mv[MU];
    const int pv = i < w ? a.piv[(int64_t)p * NB + i] : 0;
#pragma unroll
    for (int u = 0; u < MU; ++u) mv[u] = __ldg(&a.linv[(int64_t)p * NB * NB + tid + kFoldThreads * u]);
    double dv = 0.0;
    if (tid < 2 * NB) dv = a.dblk[(int64_t)p * 2 * NB + tid];
    double yv = 0.0;
    if (in && ts == 0) yv = __ldcg(&b[(int64_t)(pd.g0 + (a.full ? pv : i)) * k + c0 + c]);
    __syncthreads();
    if (tid < 2 * NB) sd[tid] = dv;                       // D's diagonal, then its sub-diagonal (se)
#pragma unroll
    for (int u = 0; u < MU; ++u) Lm[(tid + kFoldThreads * u) / NB][(tid + kFoldThreads * u) % NB] = mv[u];
    if (ts == 0) Y[i][c] = yv;
    __syncthreads();
    double s = 0.0, s1 = 0.0;
    if (a.full) {
        for (int t = ts; t <= i; t += 2 * TS) {           // Lm is zero above its diagonal
            s += Lm[i][t] * Y[t][c];
            if (t + TS < NB) s1 += Lm[i][t + TS] * Y[t + TS][c];
        }
        s += s1;
#pragma unroll
        for (int o = MC; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        __syncthreads();
        if (ts == 0) Y[i][c] = i < w ? s : 0.0;
        __syncthreads();
        double u = 0.0;
        if (in) {
            if (se[i] != 0.0) {                           // first row of a 2x2 block
                const double A = sd[i], B = se[i], C = sd[i + 1], det = A * C - B * B;
                u = (C * Y[i][c] - B * Y[i + 1][c]) / det;
            } else if (i > 0 && se[i - 1] != 0.0) {       // second row of a 2x2 block
                const double A = sd[i - 1], B = se[i - 1], C = sd[i], det = A * C - B * B;
                u = (-B * Y[i - 1][c] + A * Y[i][c]) / det;
            } else {
                u = sd[i] != 0.0 ? Y[i][c] / sd[i] : 0.0;
            }
        }
        __syncthreads();
        if (ts == 0) Y[i][c] = u;
        __syncthreads();
    }
    s = 0.0, s1 = 0.0;
    for (int t = (i / (2 * TS)) * (2 * TS) + ts; t < w; t += 2 * TS) {
        s += Lm[t][i] * Y[t][c];
        if (t + TS < NB) s1 += Lm[t + TS][i] * Y[t + TS][c];
    }
    s += s1;
#pragma unroll
    for (int o = MC; o < 8; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (in && ts == 0) b[(int64_t)(pd.g0 + pv) * k + c0 + c] = s;
}

__device__ __forceinline__ void fold_mid_any(unsigned char *smem_raw, const FoldArgs &a, int p, int chunk, double *b) {
    if (a.k == 1) fold_mid<1>(smem_raw, a, p, chunk, b);
    else if (a.k == 2) fold_mid<2>(smem_raw, a, p, chunk, b);
    else if (a.k <= 4) fold_mid<4>(smem_raw, a, p, chunk, b);
    else fold_mid<8>(smem_raw, a, p, chunk, b);
}
// columns a middle item takes, as chosen by fold_mid_any
__host__ __device__ __forceinline__ int fold_mid_cols(int k) { return k == 1 ? 1 : k == 2 ? 2 : k <= 4 ? 4 : 8; }

// Both sweeps in one cooperative launch: level by level, a bounded grid barrier between levels.
// Item q of a level goes to warp q / gridDim.x of block q % gridDim.x.  On a barrier timeout
// bar->err is set and every block returns.
template <int NC>
__global__ void __launch_bounds__(kFoldThreads, 1) k_fold_sweeps(const FoldArgs a, double *b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int k = a.k, nch = (k + NC - 1) / NC;
    const int nb = gridDim.x, q0 = (threadIdx.x >> 5) * nb + blockIdx.x, nw = kFoldWarps * nb;
    double *ws = reinterpret_cast<double *>(smem_raw) + (threadIdx.x >> 5) * 16 * kFoldMaxNc;
    FoldItem it;
    if (a.full) {
        FoldLevel lv = a.lev[0];
        if (q0 < lv.tiles * 16 * nch) fold_load_fwd(a, lv, q0 % (lv.tiles * 16), it);
        for (int L = 0; L < a.nlev; ++L) {
            const int per = lv.tiles * 16;
            const FoldLevel nx = L + 1 < a.nlev ? a.lev[L + 1] : FoldLevel{0, 0, 0, 0};
            for (int q = q0; q < per * nch; q += nw) {
                if (q != q0) fold_load_fwd(a, lv, q % per, it);
                fold_fwd<NC>(it, ws, b, k, (q / per) * NC);
            }
            // the next level's entries, before the barrier
            if (q0 < nx.tiles * 16 * nch) fold_load_fwd(a, nx, q0 % (nx.tiles * 16), it);
            if (lv.tiles > 0 && !grid_barrier(a.bar, nb, a.limit)) return;
            lv = nx;
        }
    }
    {
        const int mc = fold_mid_cols(k), nm = (k + mc - 1) / mc;
        for (int q = blockIdx.x; q < a.npan * nm; q += nb) {
            __syncthreads();
            fold_mid_any(smem_raw, a, q % a.npan, q / a.npan, b);
        }
    }
    const bool wide = nch > 1;
    auto load_bwd = [&](const FoldLevel &l, int q) {
        const int e = q % (l.tiles * 16);
        if (wide) fold_load_bwd_wide(a, l, e, it);
        else fold_load_bwd(a, l, e, it);
    };
    FoldLevel lv = a.lev[a.nlev - 1];
    if (q0 < lv.tiles * 16 * nch) load_bwd(lv, q0);
    if (!grid_barrier(a.bar, nb, a.limit)) return;
    for (int L = a.nlev - 1; L >= 0; --L) {
        const int per = lv.tiles * 16;
        const FoldLevel nx = L > 0 ? a.lev[L - 1] : FoldLevel{0, 0, 0, 0};
        for (int q = q0; q < per * nch; q += nw) {
            if (q != q0) load_bwd(lv, q);
            if (wide) fold_bwd_wide<NC>(it, ws, b, k, (q / per) * NC);
            else fold_bwd<NC>(it, b, k, 0);
        }
        if (L == 0) break;
        if (q0 < nx.tiles * 16 * nch) load_bwd(nx, q0);
        if (lv.tiles > 0 && !grid_barrier(a.bar, nb, a.limit)) return;
        lv = nx;
    }
}

// one level of one sweep per launch (SS_SOLVE_PER_STEP, ss_solve_noalloc): warp = item
template <int NC>
__global__ void __launch_bounds__(kFoldThreads) k_fold_level(const FoldArgs a, int level, int backward, double *b) {
    __shared__ double s_ws[kFoldWarps * 16 * kFoldMaxNc];
    const int nch = (a.k + NC - 1) / NC;
    const FoldLevel lv = a.lev[level];
    const int64_t per = lv.tiles * 16, q = (int64_t)blockIdx.x * kFoldWarps + (threadIdx.x >> 5);
    if (q >= per * nch) return;
    FoldItem it;
    const int c0 = (int)(q / per) * NC, e = (int)(q % per);
    if (backward && nch > 1) {
        fold_load_bwd_wide(a, lv, e, it);
        fold_bwd_wide<NC>(it, s_ws + (threadIdx.x >> 5) * 16 * kFoldMaxNc, b, a.k, c0);
    } else if (backward) {
        fold_load_bwd(a, lv, e, it);
        fold_bwd<NC>(it, b, a.k, c0);
    } else {
        fold_load_fwd(a, lv, e, it);
        fold_fwd<NC>(it, s_ws + (threadIdx.x >> 5) * 16 * kFoldMaxNc, b, a.k, c0);
    }
}

// middle step of every panel: block = (panel, chunk of right-hand sides)
__global__ void __launch_bounds__(kFoldThreads) k_fold_mid(const FoldArgs a, double *b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fold_mid_any(smem_raw, a, blockIdx.x, blockIdx.y, b);
}

}  // namespace ssk
