// FP64-accurate products on the FP16 tensor cores: the probes' Gram matrices and tall
// products (Cholesky-QR of Alg. 2 step 4, Rayleigh-Ritz) and the sparse products A X and
// B X of the subspace iteration (Alg. 2 steps 3-5), by error-free splitting (Ozaki, Ogita,
// Oishi and Rump), with one scale per operand row and an exact integer sum over the whole
// reduction.
//
// Operand.  Element (row, t) of a dense operand sits at M[row * ld_row + t * ld_k]: for the
// Gram matrix G = X^T Y the operand rows are the columns of X (ld_row = 1, ld_k = ldx); for
// the product X Q the rows of X (ld_row = ldx, ld_k = 1) and the columns of Q; for the
// sparse product A X the rows of A (CSR) and the columns of X.
// Splitting.  Every operand row is scaled by a power of two fixed by its largest entry over
// the whole reduction (|x| < 2^E, em = E + 1022 is the largest biased exponent of the row);
// Y = round(x 2^(55 - E)) is a 56-bit integer whose 8 balanced base-128 digits q_0 .. q_7
// (|q_p| <= 64, exact in FP16) are the slices: x = 2^(E - 6) sum_p q_p 2^(-7p) up to
// 2^(E - 56).  The digits are cut from the FP64 bit pattern with integer arithmetic.
// Slice layout.  The reduction is cut into pieces of 32.  For 128-row tile rt and piece kc of a
// dense operand, eight 8 KB blocks of digits in the MMA's core-matrix layout (oz_offset below) at
// block index kc * nrt + rt.  A sparse operand has no slices in memory: its tiles hold a few per
// cent of entries, so the kernel clears a stage and places the digits of the (tile, piece) pair's
// entries itself, from a list of the pattern's entries sorted by pair (6 bytes an entry).
// Products.  An output tile of 128 x 64 entries takes, per piece, the 36 digit products with
// p + q <= 7 on the tensor cores into 8 FP32 accumulators D_d = sum_{p+q=d} (8 x 64 = 512
// tensor-memory columns), exact over 16 pieces: |D_d| <= 8 * 512 * 64^2 = 2^24.  Every 16
// pieces the accumulators are read out and summed as integers,
//     hi += D_0 2^21 + D_1 2^14 + D_2 2^7 + D_3,   lo += D_4 2^21 + D_5 2^14 + D_6 2^7 + D_7,
// so the result, (hi 2^28 + lo) 2^(E_a + E_b - 61), is the exact sum of the truncated digit
// expansion rounded once to FP64: its error is a few units of 2^-53 of
// K max|a_row| max|b_row| (K the reduction length).
// Pipeline.  Two shared-memory stages of one piece each (64 KB of A, 32 KB of B).  One warp issues
// bulk copies, one the MMAs, sixteen place sparse digits and read the accumulators out; mbarriers
// between them, so a stage refills as soon as its MMAs have read it and the MMAs of the next piece
// wait for nothing else.  What bounds it: the 24 merged MMAs of a piece (2,304 cycles of tensor
// pipe), the read-outs between groups (8 x 32 KB of tensor memory every 16 pieces) and, for dense
// operands, 96 KB a piece and SM out of L2.  A X at N = 16,384, k = 304 (17,312 pairs x 5 column
// tiles): 2.18 ms with one thread issuing copies and 72 MMAs a piece in turn and 1.1 GB of digit
// slices of A in memory, 1.45 ms now.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "grid_sync.cuh"
#include "tc_ptx.cuh"

namespace sstc {

constexpr int kOzSlices = 8;
constexpr int kOzK = 32;                              // piece width along the reduction
constexpr uint32_t kOzBlock = 128 * kOzK * 2;         // one slice block: 128 rows x 32 K, FP16
constexpr uint32_t kOzHalf = 64 * kOzK * 2;           // its 64-row half
constexpr uint32_t kOzStageA = kOzSlices * kOzBlock;  // 64 KB
constexpr uint32_t kOzStageB = kOzSlices * kOzHalf;   // 32 KB
constexpr int kOzWorkers = 512;                       // threads that place sparse digits and read out
constexpr int kOzThreads = kOzWorkers + 64;           // and the copy and MMA warps
constexpr int kOzReadEvery = 16;                      // pieces per exact FP32 accumulation
constexpr size_t kOzGemmSmem = 1024 + 2 * (size_t)(kOzStageA + kOzStageB);
constexpr unsigned long long kOzWaitNs = 1000000000ull;   // a wait gives up after this long
constexpr uint32_t kTmemColsOz = 512;                 // 8 accumulators x 64 columns

// Byte offset of element (row, k) of an R x 32 FP16 tile: 8 x 8 core matrices of 16-byte
// rows, no swizzle; 4 K-adjacent core matrices 128 bytes apart, 8-row groups 512 bytes apart.
__host__ __device__ __forceinline__ uint32_t oz_offset(int row, int k) {
    return (uint32_t)((row >> 3) * 512 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// descriptor of an R x 32 tile in that layout (leading byte offset 128, stride 512)
__device__ __forceinline__ uint64_t oz_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)(128 >> 4) << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;     // descriptor version of the sm_100 family; layout type 0 = no swizzle
    return d;
}

struct OzOperand {
    const double *M;
    int64_t ld_row, ld_k;
    int64_t rows, kdim;
    const double *kscale = nullptr;                   // element (row, t) times kscale[t] (null: 1)
    __device__ __forceinline__ double at(int64_t row, int64_t t) const {
        const double v = M[row * ld_row + t * ld_k];
        return kscale ? v * kscale[t] : v;
    }
};

// the 8 balanced base-128 digits (top first) of round(x 2^(55 - E)), |x| < 2^E
__device__ __forceinline__ void oz_digits(double x, int E, int (&q)[kOzSlices]) {
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7ff);
    long long y = 0;
    if (ex != 0) {
        const long long m = (bits & ((1ll << 52) - 1)) | (1ll << 52);
        const int sh = ex - 1020 - E;                 // y = m 2^sh, sh <= 2
        if (sh >= 0) y = m << sh;
        else if (sh > -60) y = (m + (1ll << (-sh - 1))) >> (-sh);
        if (bits < 0) y = -y;
    }
#pragma unroll
    for (int p = kOzSlices - 1; p > 0; --p) {
        int d = (int)(y & 127);
        if (d >= 64) d -= 128;
        q[p] = d;
        y = (y - d) >> 7;
    }
    q[0] = (int)y;                                    // |y| < 2^55: |q_0| <= 64
}

__device__ __forceinline__ int biased_exp(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7ff); }

// em[row] = max(em[row], largest biased exponent of the row over reduction range
// [blockIdx.y per_k, (blockIdx.y + 1) per_k)); em zeroed by the caller.  Thread = row.
__global__ void __launch_bounds__(128) k_oz_expmax(OzOperand op, int64_t per_k, int *__restrict__ em) {
    const int64_t row = (int64_t)blockIdx.x * 128 + threadIdx.x;
    if (row >= op.rows) return;
    const int64_t t0 = (int64_t)blockIdx.y * per_k, t1 = min(op.kdim, t0 + per_k);
    int m = 0;
#pragma unroll 8
    for (int64_t t = t0; t < t1; ++t) m = max(m, biased_exp(op.at(row, t)));
    if (m > 0) atomicMax(&em[row], m);
}

// em[row] = largest biased exponent of CSR row `row` (0 for an empty or zero row); one warp per row
__global__ void __launch_bounds__(256) k_oz_csr_expmax(int64_t n, const int64_t *__restrict__ rowptr,
                                                       const double *__restrict__ vals, int *__restrict__ em) {
    const int64_t row = (blockIdx.x * 256ll + threadIdx.x) >> 5;
    if (row >= n) return;
    int m = 0;
    for (int64_t p = rowptr[row] + (threadIdx.x & 31); p < rowptr[row + 1]; p += 32) m = max(m, biased_exp(vals[p]));
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) em[row] = m;
}

// Block (rt, kc), thread = row of the tile and every NT / 128-th chunk of 8 columns.  Zero
// rows / columns pad the operand.  With few blocks a load's latency is the limit: 512 threads (N = 5,280,
// k = 112: dense products 16.4 -> 13.7 ms a window); with many, 128 threads write the wider runs
// (N = 16,384, k = 304: both products of a step 0.63 ms, 0.66 with 512).
template <int NT>
__global__ void __launch_bounds__(NT) k_oz_slice(OzOperand op, const int *__restrict__ em,
                                                 unsigned char *__restrict__ sl) {
    const int rt = blockIdx.x, kc = blockIdx.y;
    const int nrt = gridDim.x;
    const int rho = threadIdx.x % 128;
    const int64_t row = (int64_t)rt * 128 + rho;
    const int64_t t0 = (int64_t)kc * kOzK;
    const bool live = row < op.rows;
    const int E = (live ? em[row] : 0) - 1022;
    unsigned char *blk = sl + ((uint64_t)kc * nrt + rt) * kOzStageA;
    for (int c = threadIdx.x / 128; c < kOzK / 8; c += NT / 128) {
        __align__(16) __half h[kOzSlices][8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t t = t0 + 8 * c + u;
            const double v = (live && t < op.kdim) ? op.at(row, t) : 0.0;
            int q[kOzSlices];
            oz_digits(v, E, q);
#pragma unroll
            for (int p = 0; p < kOzSlices; ++p) h[p][u] = __int2half_rn(q[p]);   // |q| <= 64: exact
        }
#pragma unroll
        for (int p = 0; p < kOzSlices; ++p)
            *reinterpret_cast<uint4 *>(blk + (uint64_t)p * kOzBlock + oz_offset(rho, 8 * c)) =
                *reinterpret_cast<const uint4 *>(h[p]);
    }
}

struct OzMM {
    const unsigned char *slA;    // dense A: slices (null: sparse A)
    const int *emA;
    int nrtA;
    int64_t rowsA;
    const int32_t *tile_ptr;     // sparse A: pairs of row tile rt are [tile_ptr[rt], tile_ptr[rt + 1])
    const int32_t *pair_piece;   // reduction piece of pair q
    const int64_t *ent_ptr;      // entries of pair q are [ent_ptr[q], ent_ptr[q + 1])
    const uint32_t *ent_e;       // CSR position minus rowptr[128 rt]
    const uint16_t *ent_off;     // oz_offset of the entry in its block
    const int64_t *rowptr;
    const double *vals;
    const unsigned char *slB;
    const int *emB;
    int nrtB;
    int64_t rowsB;
    int nkc, per;                // dense A: pieces [z per, min(nkc, (z + 1) per)), block kc * nrtA + rt
    int mode;                    // 0: out += alpha r (atomic); 1: out = alpha s_col r + beta out;
                                 // 2: sampled (dense A): CTA x is output tile (samp_rt[x], samp_ct[x]) and
                                 // writes alpha r of its entries to out
    const int32_t *samp_rt, *samp_ct;
    const int64_t *samp_ptr;     // entries of tile x are [samp_ptr[x], samp_ptr[x + 1])
    const uint32_t *samp_e, *samp_t;   // CSR position of the entry and of its mirror image
    const uint16_t *samp_off;    // 64 (row in the tile) + column in the tile
    double alpha, beta;
    const double *colscale;      // mode 1: per-column factor s_col (null: 1)
    double *out;
    int64_t ldo;
    int *status;                 // raised when a bounded wait runs out
};

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// wait for a phase; false (and *ok cleared) after kOzWaitNs, or when another role has given up
__device__ __forceinline__ bool oz_wait(uint64_t *bar, uint32_t parity, volatile int *ok) {
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0u) {
            if (!*ok) return false;
            const unsigned long long t = gb_clock_ns();
            if (t0 == 0) t0 = t;
            else if (t - t0 > kOzWaitNs) {
                *ok = 0;
                return false;
            }
        }
    }
}

// Output tile (rt, bj) = rows 128 rt .., columns 64 bj ..  (beta = 0 does not read out).
// blockIdx.x = bj varies fastest, so the CTAs that share one A tile run together.  Worker warp w
// reads tensor-memory lanes 32 (w mod 4) .. + 31 and columns 16 (w / 4) .. + 15.
__global__ void __launch_bounds__(kOzThreads, 1) k_oz_mm(const OzMM g) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *stage[2];         // A digits, then B digits
    stage[0] = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    stage[1] = stage[0] + kOzStageA + kOzStageB;
    // full: copies landed; placed: sparse digits written (half of the worker warps); empty: MMAs of the stage
    // done; accfull: accumulators complete; accfree: read out (worker warps)
    __shared__ __align__(8) uint64_t full[2], placed[2], empty[2], accfull, accfree, drain;
    __shared__ uint32_t s_tmem;
    __shared__ int s_ok, s_em[128];
    const bool sampled = g.mode == 2;
    const int bj = sampled ? g.samp_ct[blockIdx.x] : blockIdx.x, rt = sampled ? g.samp_rt[blockIdx.x] : blockIdx.y;
    const bool sparse = g.slA == nullptr;
    int q0, q1;
    if (sparse) {
        q0 = g.tile_ptr[rt];
        q1 = g.tile_ptr[rt + 1];
    } else {
        q0 = blockIdx.z * g.per;
        q1 = min(g.nkc, q0 + g.per);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
    const int quarter = warp & 3, grp = (warp >> 2) & 3;
    const int64_t row = (int64_t)rt * 128 + 32 * quarter + lane;
    const int64_t col0 = (int64_t)bj * 64 + 16 * grp;
    if (q0 >= q1) {                  // no entries in this tile's rows: the product is zero
        if (g.mode == 1 && row < g.rowsA && warp < kOzWorkers / 32)
            for (int c = 0; c < 16; ++c) {
                const int64_t col = col0 + c;
                if (col >= g.rowsB) break;
                double *o = g.out + row * g.ldo + col;
                *o = g.beta != 0.0 ? g.beta * *o : 0.0;
            }
        return;
    }
    if (warp == 0) {
        tmem_alloc(&s_tmem, kTmemColsOz);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&full[b], 1);
            mbar_init(&placed[b], kOzWorkers / 64);
            mbar_init(&empty[b], 1);
        }
        mbar_init(&accfull, 1);
        mbar_init(&accfree, kOzWorkers / 32);
        mbar_init(&drain, 1);
        fence_mbar_init();
        s_ok = 1;
    }
    if (sparse && tid < 128) s_em[tid] = (int64_t)rt * 128 + tid < g.rowsA ? g.emA[(int64_t)rt * 128 + tid] : 0;
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int np = q1 - q0;
    volatile int *ok = &s_ok;
    if (warp == kOzWorkers / 32) {                                   // ---- copies
        if (lane == 0) {
            int sent = 0;
            for (int i = 0; i < np; ++i) {
                const int b = i & 1, q = q0 + i;
                if (i >= 2 && !oz_wait(&empty[b], (uint32_t)(((i >> 1) - 1) & 1), ok)) break;
                const int kc = sparse ? g.pair_piece[q] : q;
                const unsigned char *gb =
                    g.slB + ((uint64_t)kc * g.nrtB + (bj >> 1)) * kOzStageA + (uint64_t)(bj & 1) * kOzHalf;
                mbar_arrive_expect_tx(&full[b], sparse ? kOzStageB : kOzStageA + kOzStageB);
                if (!sparse) bulk_g2s(stage[b], g.slA + ((uint64_t)kc * g.nrtA + rt) * kOzStageA, kOzStageA, &full[b]);
                for (int p = 0; p < kOzSlices; ++p)
                    bulk_g2s(stage[b] + kOzStageA + p * kOzHalf, gb + (uint64_t)p * kOzBlock, kOzHalf, &full[b]);
                sent = i + 1;
            }
            // copies in flight land before the CTA may leave
            for (int i = max(0, sent - 2); i < sent; ++i)
                mbar_wait_bounded(&full[i & 1], (uint32_t)((i >> 1) & 1), 1ll << 24);
        }
    } else if (warp == kOzWorkers / 32 + 1) {                            // ---- MMAs
        if (lane == 0) {
            const uint32_t idesc = idesc_f16_f32(128, 0);
            bool fine = true;
            for (int i = 0; i < np && fine; ++i) {
                const int b = i & 1;
                fine = oz_wait(&full[b], (uint32_t)((i >> 1) & 1), ok) &&
                       (!sparse || oz_wait(&placed[b], (uint32_t)((i >> 1) & 1), ok));
                if (fine && i > 0 && i % kOzReadEvery == 0)     // the accumulators have been read out
                    fine = oz_wait(&accfree, (uint32_t)((i / kOzReadEvery - 1) & 1), ok);
                if (!fine) break;
                tc_fence_after();
                uint32_t sa_addr = smem_u32(stage[b]), sb_addr = sa_addr + kOzStageA;
                asm volatile("" : "+r"(sa_addr), "+r"(sb_addr));   // keep the descriptors per piece
                const uint64_t da = oz_desc(sa_addr), db = oz_desc(sb_addr);
#pragma unroll 1
                for (int kk = 0; kk < 2; ++kk)         // K steps of 16: two core matrices, 256 bytes
                    issue_digit_step<kOzSlices>(tmem, da + (uint64_t)(kk * (256 >> 4)), db + (uint64_t)(kk * (256 >> 4)),
                                                kOzBlock, kOzHalf, idesc, kk == 0 && i % kOzReadEvery == 0);
                mma_commit(&empty[b]);
                if (i % kOzReadEvery == kOzReadEvery - 1 || i + 1 == np) mma_commit(&accfull);
            }
            mma_commit(&drain);                        // no MMA in flight when the CTA leaves
            mbar_wait_bounded(&drain, 0, 1ll << 24);
        }
    } else {                                           // ---- sparse digits, read-out
        long long hi[16], lo[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            hi[c] = 0;
            lo[c] = 0;
        }
        auto wait = [&](uint64_t *bar, uint32_t parity) { return __all_sync(0xffffffffu, oz_wait(bar, parity, ok)) != 0; };
        auto read_out = [&](int group) -> bool {
            if (!wait(&accfull, (uint32_t)(group & 1))) return false;
            tc_fence_after();
            const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(16 * grp);
#pragma unroll
            for (int d = 0; d < kOzSlices; ++d) {
                float r[16];
                tmem_ld16(lane_base + (uint32_t)(d * 64), r);
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const long long x = (long long)__float2int_rn(r[c]) << (7 * (3 - (d & 3)));
                    if (d < 4) hi[c] += x;
                    else lo[c] += x;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&accfree);
            return true;
        };
        bool fine = true;
        int done = 0;                                  // accumulation groups read out
        if (sparse) {
            // Half of the workers fill stage 0, half stage 1, so a fill may take the time of two
            // pieces' MMAs.
            constexpr int kHalfW = kOzWorkers / 2;
            const double *vals = g.vals + g.rowptr[(int64_t)rt * 128];
            const int b = tid / kHalfW, wt = tid % kHalfW;
            unsigned char *sa = stage[b];
            auto place = [&](uint32_t o, double x) {
                int d[kOzSlices];
                oz_digits(x, s_em[(o >> 9) * 8 + ((o >> 4) & 7)] - 1022, d);
#pragma unroll
                for (int p = 0; p < kOzSlices; ++p)
                    *reinterpret_cast<__half *>(sa + (uint32_t)p * kOzBlock + o) = __int2half_rn(d[p]);
            };
            // this thread's first two entries of its next pair are loaded a fill ahead
            uint32_t off[2] = {0, 0};
            double v[2] = {0.0, 0.0};
            int64_t p1 = 0, pn = 0;
            auto ahead = [&](int q) {
                pn = g.ent_ptr[q] + wt;
                p1 = g.ent_ptr[q + 1];
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (pn + kHalfW * u < p1) {
                        off[u] = g.ent_off[pn + kHalfW * u];
                        v[u] = vals[g.ent_e[pn + kHalfW * u]];
                    }
            };
            if (b < np) ahead(q0 + b);
            for (int i = b; i < np; i += 2) {          // every worker comes to its barriers, whatever happens
                if (i >= 2 && fine) fine = wait(&empty[b], (uint32_t)(((i >> 1) - 1) & 1));
                // a group that ended with this stage's last piece is read out first: the MMAs wait
                if (fine && (done + 1) * kOzReadEvery <= i - 1) fine = read_out(done++);
                uint4 *z = reinterpret_cast<uint4 *>(sa);
#pragma unroll
                for (uint32_t o = 0; o < kOzStageA / 16; o += kHalfW) z[o + wt] = make_uint4(0, 0, 0, 0);
                asm volatile("bar.sync %0, %1;" ::"r"(1 + b), "n"(kHalfW) : "memory");
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (pn + kHalfW * u < p1) place(off[u], v[u]);
                for (int64_t p = pn + 2 * kHalfW; p < p1; p += kHalfW) place(g.ent_off[p], vals[g.ent_e[p]]);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(&placed[b]);
                if (i + 2 < np) ahead(q0 + i + 2);
                // one that ended with the other stage's last piece: this piece is ready behind it
                if (fine && (done + 1) * kOzReadEvery <= i) fine = read_out(done++);
            }
        }
        while (fine && (done + 1) * kOzReadEvery < np) fine = read_out(done++);
        if (fine) fine = read_out((np - 1) / kOzReadEvery);
        // the product rounded once; a non-finite operand row makes it NaN
        const int emA = row < g.rowsA ? g.emA[row] : 0;
        auto result = [&](int c, int64_t col) -> double {
            const int emB = g.emB[col], E = emA + emB - 2044 - 61;
            const double sc = (E >= -1022 && E <= 1023) ? __longlong_as_double((long long)(E + 1023) << 52)
                                                        : ldexp(1.0, E);
            const double r = fma(__ll2double_rn(hi[c]), 268435456.0, __ll2double_rn(lo[c])) * sc;
            return (emA == 0x7ff || emB == 0x7ff) ? __longlong_as_double(0x7ff8000000000000ll) : r;
        };
        if (sampled) {
            // the tile goes through shared memory (the stages are free: every MMA is done)
            double (*tile)[65] = reinterpret_cast<double (*)[65]>(stage[0]);
#pragma unroll
            for (int c = 0; c < 16; ++c)
                if (fine && row < g.rowsA && col0 + c < g.rowsB) tile[32 * quarter + lane][16 * grp + c] = result(c, col0 + c);
            asm volatile("bar.sync 3, %0;" ::"n"(kOzWorkers) : "memory");
            if (fine)
                for (int64_t p = g.samp_ptr[blockIdx.x] + tid; p < g.samp_ptr[blockIdx.x + 1]; p += kOzWorkers) {
                    const double v = g.alpha * tile[g.samp_off[p] >> 6][g.samp_off[p] & 63];
                    g.out[g.samp_e[p]] = v;
                    g.out[g.samp_t[p]] = v;
                }
        } else if (fine && row < g.rowsA) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int64_t col = col0 + c;
                if (col >= g.rowsB) continue;
                const double r = result(c, col);
                double *o = g.out + row * g.ldo + col;
                if (g.mode == 0) {
                    atomicAdd(o, g.alpha * r);
                } else {
                    const double s = g.colscale ? g.colscale[col] : 1.0;
                    *o = g.alpha * s * r + (g.beta != 0.0 ? g.beta * *o : 0.0);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && !s_ok) atomicExch(g.status, 1);
    if (warp == 0) tmem_dealloc(tmem, kTmemColsOz);
}

}  // namespace sstc
