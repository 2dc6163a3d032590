// Sparse kernels over the CSR pattern of A union B (FP64).
//   SpMM   Y = (alpha_j A + beta_j B) X with row-major blocks: the SpMV sweeps of the DOS
//          estimate (Section 3.1), B V of Alg. 2 step 3, and the residual A X - B X Lambda
//          that follows Alg. 2.
//   SDDMM  band-energy gradient sampled on the stored pattern.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace sss {

// ---------------------------------------------------------------- SpMM
// one warp per row, lanes over right-hand-side columns (k >= 16)
__global__ void k_spmm_cols(int64_t n, const int64_t *__restrict__ rowptr,
                            const int32_t *__restrict__ colind, const double *__restrict__ a,
                            const double *__restrict__ b, const double *__restrict__ alpha,
                            const double *__restrict__ beta, const double *__restrict__ X, int64_t ldx, int k,
                            double *__restrict__ Y, int64_t ldy) {
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const int64_t p0 = rowptr[row], p1 = rowptr[row + 1];
    for (int c0 = 0; c0 < k; c0 += 32) {
        const int c = c0 + lane;
        if (c >= k) break;
        const double al = alpha ? alpha[c] : 1.0, be = beta ? beta[c] : 0.0;
        double acc = 0.0;
        for (int64_t p = p0; p < p1; ++p) {
            double v = al * a[p] + (be != 0.0 ? be * b[p] : 0.0);
            acc += v * X[(int64_t)colind[p] * ldx + c];
        }
        Y[row * ldy + c] = acc;
    }
}

// one warp per row, every column in one pass over the row: lane l owns columns
// l, l+32, ..., NC accumulators (k <= 32 NC)
template <int NC>
__global__ void __launch_bounds__(256) k_spmm_rows(int64_t n, const int64_t *__restrict__ rowptr,
                                                   const int32_t *__restrict__ colind, const double *__restrict__ a,
                                                   const double *__restrict__ b, const double *__restrict__ alpha,
                                                   const double *__restrict__ beta, const double *__restrict__ X,
                                                   int64_t ldx, int k, double *__restrict__ Y, int64_t ldy) {
    // FP64 is the scarce unit: one FMA per (nonzero, column) for A alone, two when B
    // takes part (sums of A x and B x kept apart, combined once per row)
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const bool use_b = beta != nullptr;
    double acc_a[NC], acc_b[NC];
#pragma unroll
    for (int t = 0; t < NC; ++t) { acc_a[t] = 0.0; acc_b[t] = 0.0; }
    const int64_t p0 = rowptr[row], p1 = rowptr[row + 1];
    // the row's column indices and values are loaded 32 at a time (one per lane) and
    // broadcast, so consecutive X-row loads do not wait on each other
    for (int64_t q0 = p0; q0 < p1; q0 += 32) {
        const int cnt = (int)min((int64_t)32, p1 - q0);
        const int64_t q = q0 + lane;
        const int my_col = lane < cnt ? colind[q] : 0;
        const double my_a = lane < cnt ? a[q] : 0.0;
        const double my_b = (use_b && lane < cnt) ? b[q] : 0.0;
#pragma unroll 4
        for (int e = 0; e < cnt; ++e) {
            const int col = __shfl_sync(0xffffffffu, my_col, e);
            const double av = __shfl_sync(0xffffffffu, my_a, e);
            const double bv = __shfl_sync(0xffffffffu, my_b, e);
            const double *x = X + (int64_t)col * ldx;
#pragma unroll
            for (int t = 0; t < NC; ++t) {
                const int c = lane + 32 * t;
                if (c < k) {
                    const double xv = x[c];
                    acc_a[t] += av * xv;
                    if (use_b) acc_b[t] += bv * xv;
                }
            }
        }
    }
#pragma unroll
    for (int t = 0; t < NC; ++t) {
        const int c = lane + 32 * t;
        if (c < k) {
            const double al = alpha ? alpha[c] : 1.0;
            Y[row * ldy + c] = use_b ? al * acc_a[t] + beta[c] * acc_b[t] : al * acc_a[t];
        }
    }
}

// One warp per (row, chunk of KW columns), lanes over the row's nonzeros: the FP64 pipe (2
// multiply-adds a clock and SM) is the limit, and it gets one multiply-add per entry and column (two
// with B, the sums of A x and B x kept apart) with every lane busy whatever KW is.  Columns
// c0 = KW blockIdx.y ..; the lanes' sums, filled up with zeros to a power of two, are folded so that a
// step adds half as many values as the one before (32 lanes, 5 to 8 values: 9 additions a lane; an odd
// number of values is added whole at every step, 35 for 7).  N = 16,384 (472 entries a row), A alone:
// k = 4 216 us with al a + be b formed per entry and column, 76 us now (FP64 floor 53 us); k = 25 587 -> 434
// with the power of two; a band of 97 entries a row, k = 31 236 -> 153 with the same trips for every lane.
template <int V, int OFF>
__device__ __forceinline__ void spmm_fold(double *v, int lane, int &base, int &left, bool &owner) {
    static_assert((V & (V - 1)) == 0, "a power of two");
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
        spmm_fold<V / 2, OFF / 2>(v, lane, base, left, owner);
    } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], OFF);
        owner &= (lane & OFF) == 0;
        spmm_fold<1, OFF / 2>(v, lane, base, left, owner);
    }
}

template <int KW, bool WITH_B>
__global__ void __launch_bounds__(256, WITH_B ? 4 : 5)
k_spmm_nnz(int64_t n, const int64_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
           const double *__restrict__ a, const double *__restrict__ b, const double *__restrict__ alpha,
           const double *__restrict__ beta, const double *__restrict__ X, int64_t ldx, int k, double *__restrict__ Y,
           int64_t ldy) {
    const int64_t row = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, c0 = blockIdx.y * KW, kc = min(KW, k - c0);
    if (row >= n) return;
    constexpr int KP = KW > 4 ? 8 : KW > 2 ? 4 : KW, NV = WITH_B ? 2 * KP : KP;
    double acc[NV];
#pragma unroll
    for (int c = 0; c < NV; ++c) acc[c] = 0.0;
    const int64_t p0 = rowptr[row], p1 = rowptr[row + 1];
    // entry p of the row (zeros for a lane whose `in` is false)
    auto entry = [&](int64_t p, bool in) {
        const double av = in ? a[p] : 0.0;
        double bv = 0.0;
        if constexpr (WITH_B) bv = in ? b[p] : 0.0;
        const double *x = X + (int64_t)colind[p] * ldx + c0;
#pragma unroll
        for (int c = 0; c < KW; ++c)
            if (c < kc) {
                const double xv = in ? x[c] : 0.0;
                acc[c] += av * xv;
                if constexpr (WITH_B) acc[KP + c] += bv * xv;
            }
    };
    // Four entries a lane at a time while the row fills them for every lane, then what is left in one batch
    // of the same number for every lane: an unrolled loop over a lane's own entries parts the warp where the
    // counts differ (97 a row as slow as 193).
    int64_t q = p0 + lane;
    for (; q - lane + 128 <= p1; q += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u) entry(q + 32 * u, true);
    }
    auto rest = [&](auto trips) {
        constexpr int T = decltype(trips)::value;
#pragma unroll
        for (int u = 0; u + 1 < T; ++u) entry(q + 32 * u, true);
        entry(min(q + 32 * (T - 1), p1 - 1), q + 32 * (T - 1) < p1);
    };
    const int left_over = (int)(p1 - (q - lane));            // 0 .. 127
    if (left_over > 96) rest(std::integral_constant<int, 4>{});
    else if (left_over > 64) rest(std::integral_constant<int, 3>{});
    else if (left_over > 32) rest(std::integral_constant<int, 2>{});
    else if (left_over > 0) rest(std::integral_constant<int, 1>{});
    int base = 0, left = 0;
    bool owner = true;
    spmm_fold<NV, 16>(acc, lane, base, left, owner);
    // value v of the folded sums is A x (v < KP) or B x (v >= KP) of column c0 + v mod KP
    if constexpr (WITH_B) {
        __shared__ double s_sum[8][NV];
        double *s = s_sum[threadIdx.x >> 5];
#pragma unroll
        for (int e = 0; e < NV; ++e)
            if (e < left && owner) s[base + e] = acc[e];
        __syncwarp();
        for (int c = lane; c < kc; c += 32)
            Y[row * ldy + c0 + c] = (alpha ? alpha[c0 + c] : 1.0) * s[c] + beta[c0 + c] * s[KP + c];
    } else {
#pragma unroll
        for (int e = 0; e < NV; ++e)
            if (e < left && owner && base + e < kc)
                Y[row * ldy + c0 + base + e] = (alpha ? alpha[c0 + base + e] : 1.0) * acc[e];
    }
}

// ---------------------------------------------------------------- SDDMM gradient
// block per row r; X[r][:] (and lambda-weighted) in shared memory; warp per nonzero
__global__ void __launch_bounds__(256) k_sddmm(int64_t n, const int64_t *__restrict__ rowptr,
                                               const int32_t *__restrict__ colind,
                                               const double *__restrict__ X,
                                               const double *__restrict__ lam, int ne,
                                               double *__restrict__ ga, double *__restrict__ gb) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *xr = reinterpret_cast<double *>(smem_raw);
    double *xl = xr + ne;
    const int64_t r = blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < ne; i += 256) {
        double v = X[r * ne + i];
        xr[i] = v;
        xl[i] = v * lam[i];
    }
    __syncthreads();
    for (int64_t p = rowptr[r] + wid; p < rowptr[r + 1]; p += 8) {
        const double *xc = X + (int64_t)colind[p] * ne;
        double sa = 0.0, sb = 0.0;
        for (int i = lane; i < ne; i += 32) {
            double v = xc[i];
            sa += xr[i] * v;
            sb += xl[i] * v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            sa += __shfl_down_sync(0xffffffffu, sa, o);
            sb += __shfl_down_sync(0xffffffffu, sb, o);
        }
        if (lane == 0) {
            if (ga) ga[p] = sa;
            if (gb) gb[p] = -sb;
        }
    }
}

}  // namespace sss
