// Tensor-core Schur-complement update of the FP64 multifrontal factorisation (K3 of
// Alg. 2 step 2: F22 -= L21 W^T, W = L21 D) on the FP16 tensor cores, FP64-accurate by an
// error-free splitting of the operands (the slicing scheme of Ozaki, Ogita, Oishi and Rump,
// "Error-free transformations of matrix multiplication", Numer. Algorithms 2012).
//
// Splitting.  Each row x of L21 (or of W) is scaled by 2^-e, e the exponent with
// max |x_t| < 2^e, and cut into kSlices balanced 8-bit digits (digits8.cuh):
// x = 2^(e-7) sum_p q_p 2^(-8(p-1)) up to 2^(e-56), every |q_p| <= 128 (exact in FP16).
// Product.  sum_t x_it z_jt = 2^(e_i + f_j - 14) sum_{p,q} 2^(-8(p+q-2)) D_pq with the
// integer matrices D_pq = Q_p^A (Q_q^B)^T.  The pairs with p + q <= kSlices + 1 are kept
// (the rest lie below 2^-56 of the row scales); pairs of equal p + q share one FP32
// accumulator in tensor memory.  Over K = 64 every partial sum is an integer of magnitude
// below 7 * 64 * 128^2 < 2^23, so the FP32 accumulation is exact.
// Combination.  The accumulators are summed as one 64-bit integer in units of 2^(e_i + f_j - 56)
// (well below the dropped products) and packed into an FP64 by shifts; one FP64 addition applies it to
// the front.
//
// Data flow per factor step: k_panel writes L21 (in place) and W (scratch) in FP64;
// k_tc_slice writes their digits, already in the MMA's shared-memory layout (see
// tc_ptx.cuh), as one 16 KB block per (operand, 128-row tile, digit), and the row
// exponents; k_schur_tc's CTAs walk the 128 x 64 output tiles: one bulk copy brings
// the 7 A-digits of a row tile, seven bring the B-digits of its column half-tile, one
// thread issues the MMAs (40, see issue_digit_step), sixteen warps read the 7 accumulators back and
// update the FP64 front while the next tile's operands arrive.  Every wait is bounded; a wait that
// runs out records a timeout in the shift's counters, and the CTA still releases its tensor memory.
//
// What bounds it: the read-out of 7 x 32 KB of tensor memory a tile.  FP64 instructions run at 2 a
// clock and SM, so there is one per entry.  Digits and updates of a factorisation at N = 16,384
// (133 steps): 38.0 ms with one tile a CTA, FP64 digit cutting, FP64 conversions and two FP64
// multiply-adds an entry; 36.3 with merged MMAs alone; 15.6 now.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "digits8.cuh"
#include "factor_kernels.cuh"
#include "tc_ptx.cuh"

namespace sstc {

constexpr int kSlices = kTcSlices;
constexpr int kTileM = 128;                   // output rows per CTA (TMEM lanes)
constexpr int kTileN = 64;                    // output columns per CTA
constexpr uint32_t kSliceBytes = (uint32_t)kTcSliceBytes;   // one 128 x 64 FP16 block
constexpr uint32_t kHalfSliceBytes = 64 * 64 * 2;           // its 64-row half
constexpr int kAccum = kSlices;               // accumulators, one per p + q
constexpr uint32_t kTmemCols = 512;           // 7 x 64 columns, rounded to a power of two
constexpr size_t kSchurTcSmem = 1024 + (size_t)kSlices * kSliceBytes + (size_t)kSlices * kHalfSliceBytes;
constexpr size_t kSelftestSmem = 1024 + (size_t)kSliceBytes + kHalfSliceBytes;
constexpr int kSchurTcThreads = 512;          // 16 warps: lane quarter w % 4, 16 columns w / 4
constexpr int kTcSliceThreads = 512;
constexpr size_t kTcSliceSmem = 1024 + (size_t)kSlices * kSliceBytes;
constexpr long long kWaitLimit = 1ll << 24;   // mbarrier polls (about a second)

// ---------------------------------------------------------------- self-test
// One 128 x 64 x 64 MMA tile of FP16 operands given in the core-matrix layout (A: 128
// rows, B: 64 rows), FP32 result written row-major to D.  status[0] = 0 ok, 1 a wait ran
// out.
__global__ void __launch_bounds__(128, 1) k_tc_selftest(const unsigned char *__restrict__ A,
                                                         const unsigned char *__restrict__ B, float *D,
                                                         int *status) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sa = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);   // swizzle atoms: 1024-aligned
    unsigned char *sb = sa + kSliceBytes;
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 0) {
        tmem_alloc(&s_tmem, 64);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        s_ok = 1;
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    if (threadIdx.x == 0) {
        mbar_arrive_expect_tx(&bar[0], kSliceBytes + kHalfSliceBytes);
        bulk_g2s(sa, A, kSliceBytes, &bar[0]);
        bulk_g2s(sb, B, kHalfSliceBytes, &bar[0]);
        if (!mbar_wait_bounded(&bar[0], 0, kWaitLimit)) {
            s_ok = 0;
        } else {
            const uint32_t idesc = idesc_f16_f32(kTileM, kTileN);
            for (int kk = 0; kk < 4; ++kk)
                mma_f16(tmem, smem_desc(smem_u32(sa) + kk * kKStepBytes), smem_desc(smem_u32(sb) + kk * kKStepBytes), idesc,
                        kk > 0);
            mma_commit(&bar[1]);
            if (!mbar_wait_bounded(&bar[1], 0, kWaitLimit)) s_ok = 0;
        }
    }
    __syncthreads();
    tc_fence_after();
    if (s_ok) {
        for (int c0 = 0; c0 < kTileN; c0 += 16) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + c0, v);
            for (int i = 0; i < 16; ++i) D[(32 * warp + lane) * kTileN + c0 + i] = v[i];
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 64);
    if (threadIdx.x == 0) status[0] = s_ok ? 0 : 1;
}

// ---------------------------------------------------------------- slice producer
// Block = one 128-row tile of L21 (the first nrt tiles of a task) or of W (the next nrt);
// thread = (row, 16 columns).  The kSlices blocks of 16 KB are put together in shared memory and
// leave as one bulk copy; that staging lets one block be resident on an SM.
__global__ void __launch_bounds__(kTcSliceThreads) k_tc_slice(const StepTask *__restrict__ tasks, int32_t ntask,
                                                                 const ssk::ShiftPtrs<double> *sp) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sm = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    __shared__ int s_emax[4][kTileM];
    const ssk::ShiftPtrs<double> &s = sp[blockIdx.y];
    const int32_t tile = blockIdx.x;
    int lo = 0, hi = ntask - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (tasks[mid].sl_pre <= tile) lo = mid; else hi = mid - 1;
    }
    const StepTask tk = tasks[lo];
    const int nrt = (tk.r + kTileM - 1) / kTileM;
    const int tt = tile - tk.sl_pre;               // 0 .. 2 nrt - 1
    const bool side_b = tt >= nrt;
    const int ti = side_b ? tt - nrt : tt;
    const int rho = threadIdx.x & (kTileM - 1), tg = threadIdx.x / kTileM;
    const int i = ti * kTileM + rho;
    const bool live = i < tk.r;
    // column t of this operand's row: src + t ld
    const double *src = side_b ? s.wbuf + tk.wbuf_off + i : s.ws + tk.front_off + (int64_t)tk.k0 * tk.m + tk.k0 + tk.w + i;
    const int64_t ld = side_b ? tk.r : tk.m;
    double v[16];
    int ex[16], em = kFtZero;
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = (live && 16 * tg + u < tk.w) ? src[(16 * tg + u) * ld] : 0.0;
#pragma unroll
    for (int u = 0; u < 16; ++u) {
        ex[u] = ft_exp(v[u], 0);
        em = max(em, ex[u]);
    }
    s_emax[tg][rho] = em;
    __syncthreads();
#pragma unroll
    for (int o = 0; o < 4; ++o) em = max(em, s_emax[o][rho]);
    if (live && tg == 0) s.ex[tk.ex_off + (side_b ? tk.r : 0) + i] = em == kFtZero ? 0 : (em == kFtNan ? em : em - 1022);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        unsigned long long z[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) z[u] = ft_biased(v[8 * h + u], ex[8 * h + u], em);
        ft_store8(z, sm + core_offset(rho, 16 * tg + 8 * h), kSliceBytes);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned char *blk = s.sl + tk.sl_off + (uint64_t)((side_b ? nrt : 0) + ti) * kSlices * kSliceBytes;
        asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(blk), "r"(smem_u32(sm)),
                     "r"((uint32_t)(kSlices * kSliceBytes))
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
    }
}

// ---------------------------------------------------------------- Schur update
// Tiles of 128 x 64 (bi, bj) of the lower triangle of a task's trailing r x r block, numbered
// q = bi (bi + 1) + bj, bj <= 2 bi + 1; tile t of the launch is tile t mod ntile of shift t / ntile.
// Warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (its rows) and columns 16 (w / 4) .. + 15 of
// every accumulator.
struct SchurTile {
    int64_t front, base;       // the front, and its first trailing row / column
    int64_t ex_off, sl_off;
    int32_t m, r, bi, bj, nrt, shift;
};

__global__ void __launch_bounds__(kSchurTcThreads, 1) k_schur_tc(const StepTask *__restrict__ tasks, int32_t ntask,
                                                                 const ssk::ShiftPtrs<double> *sp, int32_t ntile,
                                                                 int32_t total) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *sa = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    unsigned char *sb = sa + kSlices * kSliceBytes;
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto decode = [&](int32_t t) {
        SchurTile d;
        d.shift = t / ntile;
        const int32_t tile = t - d.shift * ntile;
        int lo = 0, hi = ntask - 1;
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (tasks[mid].tc_pre <= tile) lo = mid; else hi = mid - 1;
        }
        const StepTask &tk = tasks[lo];
        const int q = tile - tk.tc_pre;
        int bi = (int)((sqrtf(4.0f * q + 1.0f) - 1.0f) * 0.5f);
        while ((bi + 1) * (bi + 2) <= q) ++bi;
        while (bi * (bi + 1) > q) --bi;
        d.bi = bi;
        d.bj = q - bi * (bi + 1);
        d.r = tk.r;
        d.m = tk.m;
        d.nrt = (tk.r + kTileM - 1) / kTileM;
        d.front = tk.front_off;
        d.base = tk.k0 + tk.w;
        d.ex_off = tk.ex_off;
        d.sl_off = tk.sl_off;
        return d;
    };
    auto issue_loads = [&](const SchurTile &d) {   // one thread
        const unsigned char *ga = sp[d.shift].sl + d.sl_off + (uint64_t)d.bi * kSlices * kSliceBytes;
        const unsigned char *gb = sp[d.shift].sl + d.sl_off + (uint64_t)(d.nrt + (d.bj >> 1)) * kSlices * kSliceBytes +
                                  (uint64_t)(d.bj & 1) * kHalfSliceBytes;
        mbar_arrive_expect_tx(&bar[0], kSlices * (kSliceBytes + kHalfSliceBytes));
        bulk_g2s(sa, ga, kSlices * kSliceBytes, &bar[0]);
        for (int p = 0; p < kSlices; ++p)
            bulk_g2s(sb + p * kHalfSliceBytes, gb + (uint64_t)p * kSliceBytes, kHalfSliceBytes, &bar[0]);
    };
    if (warp == 0) {
        tmem_alloc(&s_tmem, kTmemCols);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
        s_ok = 1;
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t idesc = idesc_f16_f32(kTileM, 0);
    static_assert(kAccum == kSlices && kTileN == 64, "accumulator d holds the products p + q = d");
    uint32_t phase = 0;
    SchurTile cur = decode(blockIdx.x);
    if (threadIdx.x == 0) issue_loads(cur);
    for (int32_t t = blockIdx.x; t < total; t += gridDim.x) {
        const bool more = t + (int32_t)gridDim.x < total;
        SchurTile next = cur;
        if (more) next = decode(t + gridDim.x);
        const ssk::ShiftPtrs<double> &s = sp[cur.shift];
        if (threadIdx.x == 0) {
            if (!mbar_wait_bounded(&bar[0], phase, kWaitLimit)) {
                s_ok = 0;
                mbar_wait_bounded(&bar[0], phase, kWaitLimit);         // copies in flight land
            } else {
                tc_fence_after();
#pragma unroll 1
                for (int kk = 0; kk < 4; ++kk)
                    issue_digit_step<kSlices>(tmem, smem_desc(smem_u32(sa)) + (uint64_t)(kk * (kKStepBytes >> 4)),
                                              smem_desc(smem_u32(sb)) + (uint64_t)(kk * (kKStepBytes >> 4)), kSliceBytes,
                                              kHalfSliceBytes, idesc, kk == 0);
                mma_commit(&bar[1]);
                if (!mbar_wait_bounded(&bar[1], phase, kWaitLimit)) {
                    s_ok = 0;
                    mbar_wait_bounded(&bar[1], phase, kWaitLimit);     // let MMAs in flight finish
                }
            }
            if (!s_ok) atomicAdd(&s.counts[7], 1ull);
            else if (more) issue_loads(next);                          // the operands have been read
        }
        // this thread's 16 front entries arrive meanwhile
        const int i = cur.bi * kTileM + 32 * (warp & 3) + lane, n0 = 16 * (warp >> 2), j0 = cur.bj * kTileN + n0;
        const bool some = cur.bi * kTileM + 32 * (warp & 3) < cur.r && j0 <= cur.bi * kTileM + 32 * (warp & 3) + 31;
        double *F = s.ws + cur.front + (cur.base + j0) * (int64_t)cur.m + cur.base + i;
        double cv[16];
        const int ei = (some && i < cur.r) ? s.ex[cur.ex_off + i] : 0;
        if (some) {
#pragma unroll
            for (int c = 0; c < 16; ++c) cv[c] = (i < cur.r && j0 + c <= i) ? F[c * (int64_t)cur.m] : 0.0;
        }
        phase ^= 1;
        __syncthreads();
        if (!s_ok) break;
        tc_fence_after();
        if (some) {
            const int32_t *fex = s.ex + cur.ex_off + cur.r + j0;
            long long T[16];
            ft_sum(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)n0, T);
            bool far = false;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int E = ei + ((j0 + c < cur.r) ? fex[c] : 0) - kTUnit;
                far |= (unsigned)(E + 950) > 1850u;
            }
            if (__any_sync(0xffffffffu, far)) {    // scales at the ends of the range, or non-finite
#pragma unroll 1
                for (int c = 0; c < 16; ++c) {
                    if (i >= cur.r || j0 + c > i) continue;
                    long long Tc = T[0];
                    double x = cv[0];
#pragma unroll
                    for (int u = 1; u < 16; ++u) {
                        Tc = u == c ? T[u] : Tc;
                        x = u == c ? cv[u] : x;
                    }
                    const int E = ei + fex[c] - kTUnit;
                    const double v = E >= kFtNan - 8192 ? __longlong_as_double(0x7ff8000000000000ll)
                                                        : (Tc == 0 ? 0.0 : ldexp((double)Tc, E));
                    F[c * (int64_t)cur.m] = x - v;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    T[c] = (long long)ft_pack(T[c], ei + ((j0 + c < cur.r) ? fex[c] : 0) - kTUnit);
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    if (i < cur.r && j0 + c <= i) F[c * (int64_t)cur.m] = cv[c] - __longlong_as_double(T[c]);
            }
        }
        tc_fence_before();
        __syncthreads();                           // the accumulators are free
        cur = next;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace sstc
