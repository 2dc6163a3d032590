// Block solves with the folded FP64 factor on the FP16 tensor cores (fold_kernels.cuh has the
// method and the CUDA-core form): b2 -= G b1 and x1 -= G^T x2 level by level, FP64-accurate by the
// error-free splitting of tc_kernels.cuh (7 balanced 8-bit digits a value, the 28 digit products
// p + q <= 6 into 7 FP32 accumulators that stay exact over 64 terms).
//
// An item is one 64-row tile of a panel's G times 128 right-hand sides.  Both sweeps put the
// right-hand sides on the 128 rows (tensor-memory lanes) of the MMA, so that a warp's atomics go to
// 32 neighbouring doubles of one row of the N x k block:
//   forward   D(c, i) = sum_t b1(t, c) G(i, t):  A = b1^T (128 x 64, K = t), B = G (64 rows, K-major)
//   backward  D(c, t) = sum_i x2(i, c) G(i, t):  A = x2^T (128 x 64, K = i), B = the same tile of G,
//             read along its other axis (the MN-major operand form)
// G's digits are scaled by row, after column t has been multiplied by 2^s_t (a.sc: about the square root
// of the diagonal of A - sigma B's terms).  G = F21 F11^-1 takes the factor S2 G S1^-1 when the pencil is
// scaled to S A S, S B S, so with s_t the digits do not change with the scale of the basis: badly scaled
// rows lose none of them.  Forward, b1(t) is multiplied by 2^-s_t, backward the result; in the backward
// product the row index is summed over, so the row scales 2^e_i are moved into x2 first.  All of these are
// additions to exponents.  Each right-hand-side column of an item has its own scale over the item's 64
// terms.  One front of 700 rows scaled by 2^-20 .. 2^20, 300 right-hand sides, relative error of a solve
// against 64 bits: 2.6e-6 without s_t, 6.0e-16 with it (CUDA cores 6.3e-16; unscaled 6.0e-16).
//
// Cutting and summing digits takes integer instructions only (digits8.cuh).  A non-finite operand
// makes its whole column (row) of the product NaN.
//
// What bounds it: an item's load and cut, MMAs and read-out, which take turns.  One item a level over 258
// level steps would be 2.7 ms at N = 16,384, k = 304; the rest of its 8.8 are items queued in wide levels.
// Measured per item (cycles): right-hand sides' load and digits 6,000, 40 MMAs 4,250 (7,100 as 112 MMAs of N = 64), read-out 8,100 (7 x 32 KB out
// of tensor memory), the next tile's digits 3,100, barrier 4,000-7,000; G's tile of the next level
// is loaded during the MMAs and cut before the barrier.  (Measured before the zero test moved into the
// exponent and scales came four at a time, 4% of a solve.)  One solve at N = 16,384, k = 304: 61.8 ms on the CUDA
// cores (0.87 of their FP64 peak), 8.8 ms here; N = 5,280, k = 112: 4.4 -> 1.5 ms.
// Tried and left out: an accumulator's read-out under the MMAs of the next ones (each slows the
// other: 9,000 + 8,400 cycles where one after the other takes 7,100 + 8,100).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fold_kernels.cuh"
#include "digits8.cuh"
#include "tc_ptx.cuh"

namespace sstc {

using ssk::NB;

constexpr int kFtThreads = 512;
constexpr int kFtCols = 128;                        // right-hand sides of an item
constexpr int kFtRows = 64;                         // rows of G in an item
constexpr uint32_t kFtSliceA = kFtCols * 64 * 2;    // one digit of the right-hand sides: 16 KB
constexpr uint32_t kFtSliceB = kFtRows * 64 * 2;    // one digit of G: 8 KB
constexpr size_t kFtSmem = 1024 + (size_t)kFtSlices * (kFtSliceA + kFtSliceB);
constexpr uint32_t kFtTmemCols = 512;               // 7 accumulators x 64 columns
constexpr long long kFtWaitLimit = 1ll << 24;

// Right-hand sides of an item of a level of `tiles` row tiles on nb blocks: 64 where items of 128 would
// leave half of the blocks without one (a thread then cuts 8 terms instead of 16), else 128
__host__ __device__ __forceinline__ int ft_width(int tiles, int k, int nb) {
    return 2 * tiles * ((k + kFtCols - 1) / kFtCols) <= nb ? kFtCols / 2 : kFtCols;
}
// multiply-adds' flops that the tensor cores do for an item: 28 digit products of 128 x 64 x 64
constexpr double kFtItemFlops = 28.0 * 2.0 * kFtCols * kFtRows * NB;

// The MMAs of one item: accumulator d (columns 64 d ..) = sum_{p + q = d} A_p B_q^T.  Per K step of 16
// the right-hand sides advance 32 bytes inside their 128-byte rows; G does the same when K is its
// column (forward), or 16 rows = 2,048 bytes when K is its row (backward, MN-major: the next 64 of
// a merged N, the next digit, lie a leading byte offset of 8 KB further).
__device__ __forceinline__ void ft_issue(uint32_t tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t bstep) {
#pragma unroll 1
    for (int kk = 0; kk < 4; ++kk)
        issue_digit_step<kFtSlices>(tmem, da + (uint64_t)(kk * (kKStepBytes >> 4)), db + (uint64_t)(kk * (bstep >> 4)),
                                    kFtSliceA, kFtSliceB, idesc, kk == 0);
}

__global__ void __launch_bounds__(kFtThreads, 1) k_fold_tc(const ssk::FoldArgs a, double *b) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sa = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *sb = sa + kFtSlices * kFtSliceA;
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok;
    __shared__ int s_emax[8][kFtCols], s_gmax[8][kFtRows];
    __shared__ int s_ec[kFtCols];                   // em of every right-hand-side column
    __shared__ __align__(16) int s_er[kFtRows];     // E of every row of G (|G row| < 2^E), kFtZero, kFtNan
    __shared__ int s_row[kFtRows];                  // global row of every row of G
    __shared__ __align__(16) int s_ce[NB];          // minus the scale exponent of every column of G
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k = a.k, nb = gridDim.x;
    if (warp == 0) {
        tmem_alloc(&s_tmem, kFtTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        s_ok = 1;
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t idesc_f = idesc_f16_f32(kFtCols, 0), idesc_b = idesc_f | (1u << 16);   // bit 16: B is MN-major
    const uint64_t lbo_b = (uint64_t)((kFtSliceB >> 4) - 1) << 16;   // added to the forward form's field of 1
    uint32_t phase = 0;

    // ---- the item in hand, and the one whose entries are being fetched
    ssk::FoldTile tl{};
    double g[8];                                    // G(row gi, columns 8 gt ..)
    int grow = 0;                                   // its global row
    int gce = 0;                                    // lane l: scale exponent of column 8 gt + l mod 8
    const int gi = tid & 63, gt = tid >> 6;
    auto fetch = [&](const ssk::FoldTile &t) {
        tl = t;
        const double *F = a.arena + t.off + (int64_t)(8 * gt) * t.m + gi;
        if (gt == 0 && gi < t.nr) grow = a.idx[t.idx + gi];
        gce = 8 * gt + (lane & 7) < t.w ? __ldg(a.sc + t.g0 + 8 * gt + (lane & 7)) : 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = (gi < t.nr && 8 * gt + u < t.w) ? __ldg(F + (int64_t)u * t.m) : 0.0;
    };
    // digits of the fetched tile of G into sb, its row exponents and global rows
    auto cut_g = [&]() {
        int ex[8], em = kFtZero;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            ex[u] = ft_exp(g[u], __shfl_sync(0xffffffffu, gce, u));
            em = max(em, ex[u]);
        }
        s_gmax[gt][gi] = em;
        if (gt == 0) s_row[gi] = grow;
        if (gi < 8) s_ce[8 * gt + gi] = -gce;
        __syncthreads();
#pragma unroll
        for (int o = 0; o < 8; ++o) em = max(em, s_gmax[o][gi]);
        if (gt == 0) s_er[gi] = (em == kFtZero || em == kFtNan) ? em : em - 1022;
        unsigned long long z[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = ft_biased(g[u], ex[u], em);
        ft_store8(z, sb + core_offset(gi, 8 * gt), kFtSliceB);
    };
    // Digits of the item's right-hand sides [c0, c1) into sa: terms b1(t) 2^-s_t (forward) or
    // x2(row i) 2^e_i (backward); needs s_row, s_er, s_ce of the item.  A thread cuts V terms of a column:
    // 8 where at most 64 right-hand sides exist, else 16.  Rows of the operand without a
    // right-hand side stay as they are: nothing reads those products.
    auto cut_rhs_v = [&](auto vc, int c0, int c1, bool backward, const ssk::FoldTile &t) {
        constexpr int V = decltype(vc)::value, W = kFtThreads * V / 64, G = 64 / V;   // columns, parts of a column
        const int c = tid % W, tg = tid / W;
        const bool work = c0 + (c & ~31) < c1;
        double v[V];
        int ex[V], em = kFtZero;
        if (work) {
#pragma unroll
            for (int u = 0; u < V; ++u) {
                const int n = V * tg + u;
                const bool in = c0 + c < c1 && n < (backward ? t.nr : t.w);
                const int64_t row = backward ? s_row[n] : t.g0 + n;
                v[u] = in ? __ldcg(&b[row * k + c0 + c]) : 0.0;
            }
            const int4 *sh = reinterpret_cast<const int4 *>((backward ? s_er : s_ce) + V * tg);
#pragma unroll
            for (int u = 0; u < V; u += 4) {
                const int4 h = sh[u / 4];
                ex[u] = ft_exp(v[u], h.x), ex[u + 1] = ft_exp(v[u + 1], h.y);
                ex[u + 2] = ft_exp(v[u + 2], h.z), ex[u + 3] = ft_exp(v[u + 3], h.w);
                em = max(max(em, max(ex[u], ex[u + 1])), max(ex[u + 2], ex[u + 3]));
            }
            s_emax[tg][c] = em;
        }
        __syncthreads();
        if (!work) return;
#pragma unroll
        for (int o = 0; o < G; ++o) em = max(em, s_emax[o][c]);
        if (tg == 0) s_ec[c] = em;
#pragma unroll
        for (int h = 0; h < V / 8; ++h) {
            unsigned long long z[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) z[u] = ft_biased(v[8 * h + u], min(ex[8 * h + u], em), em);
            ft_store8(z, sa + core_offset(c, V * tg + 8 * h), kFtSliceA);
        }
    };
    auto cut_rhs = [&](int c0, int c1, bool backward, const ssk::FoldTile &t) {
        if (c1 - c0 <= 64) cut_rhs_v(std::integral_constant<int, 8>{}, c0, c1, backward, t);
        else cut_rhs_v(std::integral_constant<int, 16>{}, c0, c1, backward, t);
    };
    // MMAs of the item, complete on return (false: a wait ran out)
    auto multiply = [&](bool backward) -> bool {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");    // digits visible to the tensor cores
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
            ft_issue(tmem, smem_desc(smem_u32(sa)), smem_desc(smem_u32(sb)) + (backward ? lbo_b : 0),
                     backward ? idesc_b : idesc_f, backward ? 16u * 128u : kKStepBytes);
            mma_commit(&bar);
            if (!mbar_wait_bounded(&bar, phase, kFtWaitLimit)) {
                s_ok = 0;
                mbar_wait_bounded(&bar, phase, kFtWaitLimit);           // let MMAs in flight finish
            }
        }
        phase ^= 1;
        __syncthreads();
        tc_fence_after();
        return s_ok != 0;
    };
    // Subtract the product from the N x k block: column n of the accumulators goes to row s_row[n]
    // (forward) or g0 + n (backward).  Sixteen values first, then their atomics: no branch between
    // them, so the columns' chains overlap.  Scales near the ends of the exponent range and
    // non-finite operands take the other path, which may use FP64 instructions.
    auto read_out = [&](int c0, int c1, bool backward, const ssk::FoldTile &t) {
        const int c = 32 * (warp & 3) + lane, n0 = 16 * (warp >> 2);
        if (c0 + 32 * (warp & 3) >= c1) return;      // this warp's right-hand sides do not exist
        const int ec = s_ec[c] - 1022 - kTUnit, lim = backward ? t.w : t.nr;
        const bool live = c0 + c < c1;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)n0;
        long long T[16];
        // scales of the warp's rows (forward) or columns (backward) of G; every lane needs the ends of their
        // range only
        const int *es = (backward ? s_ce : s_er) + n0;
        const int el = es[lane & 15];
        const int emax = __reduce_max_sync(0xffffffffu, el == kFtZero ? -(1 << 19) : el);
        const int emin = __reduce_min_sync(0xffffffffu, el == kFtZero ? 1 << 19 : el);
        // a zero column: its products are zero
        const bool far = live && s_ec[c] > kFtZero / 2 && (ec + emin < -950 || ec + emax > 900);
        ft_sum(lane_base, T);
        tc_fence_before();
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] = -T[e];
        if (__any_sync(0xffffffffu, far)) {
#pragma unroll 1
            for (int e = 0; e < 16; ++e) {
                const int n = n0 + e, ee = es[e];
                long long Te = T[0];
#pragma unroll
                for (int u = 1; u < 16; ++u) Te = u == e ? T[u] : Te;
                const double v = (ec >= kFtNan - 8192 || ee == kFtNan) ? __longlong_as_double(0x7ff8000000000000ll)
                                                                       : (Te == 0 ? 0.0 : ldexp((double)Te, ec + ee));
                const int64_t row = backward ? t.g0 + n : s_row[n];
                if (live && n < lim && v != 0.0) atomicAdd(&b[row * k + c0 + c], v);
            }
            return;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int4 v = reinterpret_cast<const int4 *>(es)[q];
            T[4 * q] = (long long)ft_pack(T[4 * q], ec + v.x);
            T[4 * q + 1] = (long long)ft_pack(T[4 * q + 1], ec + v.y);
            T[4 * q + 2] = (long long)ft_pack(T[4 * q + 2], ec + v.z);
            T[4 * q + 3] = (long long)ft_pack(T[4 * q + 3], ec + v.w);
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int n = n0 + e;
            const int64_t row = backward ? t.g0 + n : s_row[n];
            if (live && n < lim && T[e] != 0) atomicAdd(&b[row * k + c0 + c], __longlong_as_double(T[e]));
        }
    };
    auto width = [&](const ssk::FoldLevel &lv) { return ft_width(lv.tiles_64, k, nb); };
    // this block's items of a level: [qa, qb), tile fastest
    auto range = [&](const ssk::FoldLevel &lv, int &qa, int &qb) {
        const int cw = width(lv), items = lv.tiles_64 * ((k + cw - 1) / cw), per = (items + nb - 1) / nb;
        qa = min(items, (int)blockIdx.x * per);
        qb = min(items, qa + per);
    };
    auto tile = [&](const ssk::FoldLevel &lv, int q) { return a.tiles_64[lv.tile0_64 + q % lv.tiles_64]; };
    bool ok = true;
    unsigned int at = 0;
    auto sweep = [&](bool backward) {
        const int first = backward ? a.nlev - 1 : 0, step = backward ? -1 : 1;
        ssk::FoldLevel lv = a.lev[first];
        int qa, qb;
        range(lv, qa, qb);
        if (backward) ::grid_arrive(a.bar, nb, at);                                     // the middle step is done
        if (qa < qb) { fetch(tile(lv, qa)); cut_g(); }
        if (backward && !::grid_wait(a.bar, a.limit, at)) { ok = false; return; }
        for (int n = 0; n < a.nlev; ++n) {
            const bool more = n + 1 < a.nlev;
            const ssk::FoldLevel nx = more ? a.lev[first + step * (n + 1)] : ssk::FoldLevel{0, 0, 0, 0};
            int na = 0, nbq = 0;
            if (more) range(nx, na, nbq);
            if (qa == qb && na < nbq) fetch(tile(nx, na));
            const int cw = width(lv);
            int last_panel = -1, last_c0 = -1;
            for (int q = qa; q < qb; ++q) {
                const int c0 = q / lv.tiles_64 * cw, c1 = min(k, c0 + cw);
                if (q > qa) cut_g();
                const ssk::FoldTile t = tl;
                // the next item, in this level or the next: its record now, its entries during the MMAs
                const bool has = q + 1 < qb || na < nbq;
                ssk::FoldTile tn{};
                if (has) tn = q + 1 < qb ? tile(lv, q + 1) : tile(nx, na);
                __syncthreads();                     // s_row, s_er, s_ce written
                if (backward || t.g0 != last_panel || c0 != last_c0) cut_rhs(c0, c1, backward, t);
                last_panel = t.g0;
                last_c0 = c0;
                if (has) fetch(tn);
                if (!multiply(backward)) { ok = false; return; }
                read_out(c0, c1, backward, t);
                __syncthreads();                     // s_row, s_er, s_ce, s_ec and the accumulators are free
            }
            // the next item's digits while the other blocks arrive
            const bool wait = (more || !backward) && lv.tiles_64 > 0;
            if (wait) ::grid_arrive(a.bar, nb, at);
            if (na < nbq) cut_g();
            if (wait && !::grid_wait(a.bar, a.limit, at)) { ok = false; return; }
            lv = nx;
            qa = na;
            qb = nbq;
        }
    };
    if (a.full) sweep(false);
    if (ok) {
        const int mc = ssk::fold_mid_cols(k, a.npan, nb), nm = (k + mc - 1) / mc;
        for (int q = blockIdx.x; q < a.npan * nm; q += nb) {
            __syncthreads();
            ssk::fold_mid_load(sa, a, q % a.npan);
            __syncthreads();
            ssk::fold_mid_any(sa, a, mc, q % a.npan, q / a.npan, b);
        }
        __syncthreads();
        sweep(true);
    }
    if (!ok && tid == 0 && s_ok == 0) ::grid_fail(a.bar);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kFtTmemCols);
}

}  // namespace sstc
