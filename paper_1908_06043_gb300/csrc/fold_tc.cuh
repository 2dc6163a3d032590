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
// G's digits are scaled by row; in the backward product the row index is summed over, so the row
// scales 2^e_i are moved into x2 first (an exponent addition).  Each right-hand-side column of an
// item has its own scale over the item's 64 terms.
//
// Digits without conversions: y = round(x 2^(55 - E)) plus the constant 0x80..80 has the digits,
// biased by 128, as its bytes; a byte u is the FP16 number (0x6400 | u) - 1152 (one byte
// permutation, one logic operation and one packed subtraction for two digits).  The read-out
// forms the 7 accumulators' sum as one 64-bit integer (its last bits, 2^-62 of the scales, lie
// below the dropped digit products) and packs it into an FP64 by shifts: FP64 instructions run at
// 2 a clock and SM here, and an item uses none.  A non-finite operand makes its whole column (row)
// of the product NaN.
//
// What bounds it: the chain of one item a level.  Measured per item (cycles): right-hand sides'
// load and digits 6,000, 40 MMAs 4,250 (7,100 as 112 MMAs of N = 64), read-out 8,100 (7 x 32 KB out
// of tensor memory), the next tile's digits 3,100, barrier 4,000-7,000; G's tile of the next level
// is loaded during the MMAs and cut before the barrier.  One solve at N = 16,384, k = 304: 61.8 ms
// on the CUDA cores (0.87 of their FP64 peak), 9.2 ms here; N = 5,280, k = 112: 4.4 -> 1.6 ms.
// Tried and left out: an accumulator's read-out under the MMAs of the next ones (each slows the
// other: 9,000 + 8,400 cycles where one after the other takes 7,100 + 8,100).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fold_kernels.cuh"
#include "tc_ptx.cuh"

namespace sstc {

using ssk::NB;

constexpr int kFtThreads = 512;
constexpr int kFtCols = 128;                        // right-hand sides of an item
constexpr int kFtRows = 64;                         // rows of G in an item
constexpr int kFtSlices = 7;
constexpr uint32_t kFtSliceA = kFtCols * 64 * 2;    // one digit of the right-hand sides: 16 KB
constexpr uint32_t kFtSliceB = kFtRows * 64 * 2;    // one digit of G: 8 KB
constexpr size_t kFtSmem = 1024 + (size_t)kFtSlices * (kFtSliceA + kFtSliceB);
constexpr uint32_t kFtTmemCols = 512;               // 7 accumulators x 64 columns
constexpr int kFtNan = 1 << 20;                     // "exponent" of a non-finite value
constexpr int kFtZero = -(1 << 20);                 // "exponent" of zero
constexpr long long kFtWaitLimit = 1ll << 24;

// biased exponent of v plus sh; kFtZero for zero (and denormals, which count as zero), kFtNan
__device__ __forceinline__ int ft_exp(double v, int sh) {
    const int ex = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
    return ex == 0 ? kFtZero : (ex == 0x7ff ? kFtNan : ex + sh);
}

// round(x 2^(55 - E)) + 0x80808080808080 for |x| < 2^E; em = E + 1022 >= ex, the exponents as from
// ft_exp
__device__ __forceinline__ unsigned long long ft_biased(double v, int ex, int em) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    unsigned long long m = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    m = (((m << 3) >> min(em - ex, 60)) + 1) >> 1;  // 4 m 2^(ex - em), rounded
    if (ex == kFtZero) m = 0;
    const unsigned long long s = (unsigned long long)((long long)bits >> 63);
    return ((m ^ s) - s) + 0x80808080808080ull;
}

// the 7 digits of 8 values (biased as above) as FP16, 16 bytes to each slice
__device__ __forceinline__ void ft_store8(const unsigned long long (&z)[8], unsigned char *dst, uint32_t stride) {
    const __half2 bias = __half2half2(__ushort_as_half((unsigned short)0x6480));    // 1152
#pragma unroll
    for (int p = 0; p < kFtSlices; ++p) {
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const unsigned long long z0 = z[2 * e], z1 = z[2 * e + 1];
            uint32_t h;
            if (p == 0) {                           // the top digit is 0 .. 256: both bytes
                h = __byte_perm((uint32_t)(z0 >> 32), (uint32_t)(z1 >> 32), 0x7632) | 0x64006400u;
            } else {
                const int byte = 6 - p;             // of the 8 bytes of z
                const uint32_t w0 = (uint32_t)(byte >= 4 ? z0 >> 32 : z0), w1 = (uint32_t)(byte >= 4 ? z1 >> 32 : z1);
                const uint32_t b = byte & 3;
                h = (__byte_perm(w0, w1, b | (b << 4) | ((4 + b) << 8) | ((4 + b) << 12)) & 0x00ff00ffu) | 0x64006400u;
            }
            const __half2 d = __hsub2(*reinterpret_cast<const __half2 *>(&h), bias);
            o[e] = *reinterpret_cast<const uint32_t *>(&d);
        }
        *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

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

// 16 columns of one accumulator; the values are there after ft_tmem_wait on the same registers
__device__ __forceinline__ void ft_tmem_ld(uint32_t t, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(t)
        : "memory");
}
__device__ __forceinline__ void ft_tmem_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// integer-valued |a| <= 2^22 plus 0x4B400000 as an integer: the bits of a + 1.5 2^23
constexpr long long kFtMagic = 0x4B400000ll;
__device__ __forceinline__ long long ft_int22(uint32_t a) {
    return (long long)__float_as_int(__uint_as_float(a) + 12582912.0f);
}
// integer-valued |a| < 2^23 as int
__device__ __forceinline__ int ft_int23(uint32_t a) {
    const int b = (int)a, s = b >> 31;
    const int m = __float_as_int(__uint_as_float(a) + __int_as_float((b & (int)0x80000000) | 0x4B000000)) & 0x7fffff;
    return (m ^ s) - s;
}

// bits of T 2^E, rounded to nearest (ties away), by shifts and an integer addition: no branch, for
// |T| < 2^62 and results in the normal range (or T = 0)
__device__ __forceinline__ unsigned long long ft_pack(long long T, int E) {
    const unsigned long long s = (unsigned long long)(T >> 63);
    unsigned long long u = ((unsigned long long)T ^ s) - s;
    const int lz = __clzll((long long)u);           // 64 for T = 0: u stays 0
    u <<= (lz & 63);
    const unsigned long long bits = ((unsigned long long)(uint32_t)(1023 + 62 - lz + E) << 52) + (u >> 11) + ((u >> 10) & 1);
    return T == 0 ? 0ull : (bits | (s & (1ull << 63)));
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
    __shared__ int s_er[kFtRows];                   // E of every row of G (|G row| < 2^E), kFtZero, kFtNan
    __shared__ int s_row[kFtRows];                  // global row of every row of G
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
    const int gi = tid & 63, gt = tid >> 6;
    auto fetch = [&](const ssk::FoldTile &t) {
        tl = t;
        const double *F = a.arena + t.off + (int64_t)(8 * gt) * t.m + gi;
        if (gt == 0 && gi < t.nr) grow = a.idx[t.idx + gi];
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = (gi < t.nr && 8 * gt + u < t.w) ? __ldg(F + (int64_t)u * t.m) : 0.0;
    };
    // digits of the fetched tile of G into sb, its row exponents and global rows
    auto cut_g = [&]() {
        int ex[8], em = kFtZero;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            ex[u] = ft_exp(g[u], 0);
            em = max(em, ex[u]);
        }
        s_gmax[gt][gi] = em;
        if (gt == 0) s_row[gi] = grow;
        __syncthreads();
#pragma unroll
        for (int o = 0; o < 8; ++o) em = max(em, s_gmax[o][gi]);
        if (gt == 0) s_er[gi] = (em == kFtZero || em == kFtNan) ? em : em - 1022;
        unsigned long long z[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = ft_biased(g[u], ex[u], em);
        ft_store8(z, sb + core_offset(gi, 8 * gt), kFtSliceB);
    };
    // Digits of the item's right-hand sides [c0, c1) into sa: terms b1(t) (forward) or
    // x2(row i) 2^e_i (backward); needs s_row, s_er of the item.  A thread cuts V terms of a column:
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
#pragma unroll
            for (int u = 0; u < V; ++u) {
                ex[u] = ft_exp(v[u], backward ? s_er[V * tg + u] : 0);
                em = max(em, ex[u]);
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
        const int ec = s_ec[c] - 1022 - 52, lim = backward ? t.w : t.nr;
        const bool live = c0 + c < c1;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)n0;
        uint32_t r[16];
        long long T[16];
        auto load = [&](int d) {
            ft_tmem_ld(lane_base + (uint32_t)d * 64, r);
            ft_tmem_wait(r);
        };
        bool far = false;
        if (!backward) {
#pragma unroll
            for (int n = 0; n < 16; ++n) {
                const int er = s_er[n0 + n];
                far |= er != kFtZero && (ec + er < -950 || ec + er > 900);
            }
        } else {
            far = ec < -950 || ec > 900;
        }
        far &= live && s_ec[c] > kFtZero / 2;        // a zero column: its products are zero
        // T = a_0 2^38 + a_1 2^30 + a_2 2^22 + a_3 2^14 + a_4 2^6 + (a_5 2^8 + a_6) 2^-10: the magic
        // numbers' share is taken off once; the last term is rounded to FP32 (below 0.2) and to an
        // integer
        load(6);
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] = r[e];
        load(5);
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float x = fmaf(__uint_as_float(r[e]), 256.0f, __uint_as_float((uint32_t)T[e]));
            T[e] = __float_as_int(fmaf(x, 1.0f / 1024.0f, 12582912.0f));
        }
        load(4);
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] += (long long)ft_int23(r[e]) * 64;
        load(3);
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) * (1 << 14);
        load(2);
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) * (1 << 22);
        load(1);
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] += ft_int22(r[e]) * (1 << 30);
        load(0);
        tc_fence_before();
        constexpr long long kAll =
            (long long)((unsigned long long)kFtMagic * (1ull + (1ull << 14) + (1ull << 22) + (1ull << 30) + (1ull << 38)));
#pragma unroll
        for (int e = 0; e < 16; ++e)
            T[e] = kAll - (long long)((unsigned long long)T[e] + ((unsigned long long)ft_int22(r[e]) << 38));
        if (__any_sync(0xffffffffu, far)) {
#pragma unroll 1
            for (int e = 0; e < 16; ++e) {
                const int n = n0 + e, er = backward ? 0 : s_er[n];
                long long Te = T[0];
#pragma unroll
                for (int u = 1; u < 16; ++u) Te = u == e ? T[u] : Te;
                const double v = (ec >= kFtNan - 8192 || er == kFtNan) ? __longlong_as_double(0x7ff8000000000000ll)
                                                                       : (Te == 0 ? 0.0 : ldexp((double)Te, ec + er));
                const int64_t row = backward ? t.g0 + n : s_row[n];
                if (live && n < lim && v != 0.0) atomicAdd(&b[row * k + c0 + c], v);
            }
            return;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) T[e] = (long long)ft_pack(T[e], ec + (backward ? 0 : s_er[n0 + e]));
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const int n = n0 + e;
            const int64_t row = backward ? t.g0 + n : s_row[n];
            if (live && n < lim && T[e] != 0) atomicAdd(&b[row * k + c0 + c], __longlong_as_double(T[e]));
        }
    };
    // Right-hand sides of an item of a level: 64 where items of 128 would leave half of the blocks
    // without one (a thread then cuts 8 terms instead of 16), else 128
    auto width = [&](const ssk::FoldLevel &lv) {
        return 2 * lv.tiles_64 * ((k + kFtCols - 1) / kFtCols) <= nb ? kFtCols / 2 : kFtCols;
    };
    // this block's items of a level: [qa, qb), tile fastest
    auto range = [&](const ssk::FoldLevel &lv, int &qa, int &qb) {
        const int cw = width(lv), items = lv.tiles_64 * ((k + cw - 1) / cw), per = (items + nb - 1) / nb;
        qa = min(items, (int)blockIdx.x * per);
        qb = min(items, qa + per);
    };
    auto tile = [&](const ssk::FoldLevel &lv, int q) { return a.tiles_64[lv.tile0_64 + q % lv.tiles_64]; };
    bool ok = true;
    auto sweep = [&](bool backward) {
        const int first = backward ? a.nlev - 1 : 0, step = backward ? -1 : 1;
        ssk::FoldLevel lv = a.lev[first];
        int qa, qb;
        range(lv, qa, qb);
        if (qa < qb) { fetch(tile(lv, qa)); cut_g(); }
        if (backward && !::grid_barrier(a.bar, nb, a.limit)) { ok = false; return; }    // the middle step is done
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
                __syncthreads();                     // s_row, s_er written
                if (backward || t.g0 != last_panel || c0 != last_c0) cut_rhs(c0, c1, backward, t);
                last_panel = t.g0;
                last_c0 = c0;
                if (has) fetch(tn);
                if (!multiply(backward)) { ok = false; return; }
                read_out(c0, c1, backward, t);
                __syncthreads();                     // s_row, s_er, s_ec and the accumulators are free
            }
            if (na < nbq) cut_g();
            if ((more || !backward) && lv.tiles_64 > 0 && !::grid_barrier(a.bar, nb, a.limit)) { ok = false; return; }
            lv = nx;
            qa = na;
            qb = nbq;
        }
    };
    if (a.full) sweep(false);
    if (ok) {
        const int mc = ssk::fold_mid_cols(k), nm = (k + mc - 1) / mc;
        for (int q = blockIdx.x; q < a.npan * nm; q += nb) {
            __syncthreads();
            ssk::fold_mid_any(sa, a, q % a.npan, q / a.npan, b);
        }
        __syncthreads();
        sweep(true);
    }
    if (!ok && tid == 0 && s_ok == 0) atomicExch(&a.bar->err, 1);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kFtTmemCols);
}

}  // namespace sstc
