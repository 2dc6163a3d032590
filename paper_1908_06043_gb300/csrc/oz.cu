// Host side of the FP64-accurate tensor-core products (tc_gemm.cuh): operand slicing, the
// (tile, piece) plan of the sparse pattern, and the launches.
#include <algorithm>
#include <atomic>
#include <memory>
#include <mutex>
#include <new>
#include <vector>

#include "internal.h"
#include "tc_gemm.cuh"

struct OzPlan {
    int32_t nrt = 0;
    int64_t npairs = 0;
    int32_t *d_tile_ptr = nullptr, *d_pair_piece = nullptr;
    int64_t *d_ent_ptr = nullptr;      // npairs + 1
    uint32_t *d_ent_e = nullptr;       // nnz, sorted by pair
    uint16_t *d_ent_off = nullptr;
};

// entries at or below the diagonal by (128-row tile, 64-column tile), for the sampled product X Y^T:
// the tiles are counted first, the lists made by the first product that takes them
struct OzSamples {
    int64_t ntiles = 0;
    std::vector<int32_t> rts, cts;     // row and column tile of every tile (host, until the lists are made)
    std::vector<int64_t> ptr, first;   // first entry of every tile; first tile of every row tile
    int32_t *d_rt = nullptr, *d_ct = nullptr;
    int64_t *d_ptr = nullptr;          // ntiles + 1
    uint32_t *d_e = nullptr, *d_t = nullptr;   // CSR positions of the entry and its mirror image
    uint16_t *d_off = nullptr;
};

struct OzVals {
    const double *vals = nullptr;
    int *em = nullptr;                 // per row: largest biased exponent
};

namespace {

using sstc::OzOperand;

inline unsigned cdivu(int64_t a, int64_t b) { return (unsigned)((a + b - 1) / b); }

// FP16 MMA work of one (output tile, piece): 36 digit products x 2 K steps of 128 x 64 x 16
constexpr double kPieceTensorFlops = 36.0 * 2.0 * 2.0 * 128 * 64 * 16;

// per-call device scratch from the stream-ordered pool
struct Scratch {
    std::vector<void *> ptrs;
    ss_ctx *ctx;
    cudaStream_t st;
    explicit Scratch(ss_ctx *c) : ctx(c), st(c->stream) {}
    template <typename T>
    cudaError_t get(T **p, size_t count) {
        cudaError_t e = ss_malloc_async(ctx, (void **)p, sizeof(T) * std::max<size_t>(count, 1), st);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
    ~Scratch() {
        for (void *p : ptrs) cudaFreeAsync(p, st);
    }
};

#define OZ_ALLOC(ctx, expr)                                                                               \
    do {                                                                                                  \
        cudaError_t e_ = (expr);                                                                          \
        if (e_ != cudaSuccess) {                                                                          \
            cudaGetLastError();                                                                           \
            return (ctx)->set_error(SS_ERR_OOM, std::string("device allocation failed: ") +             \
                                                    cudaGetErrorString(e_));                              \
        }                                                                                                 \
    } while (0)

void oz_attrs(int device) {
    static std::mutex mu;
    static std::vector<char> seen;
    std::lock_guard<std::mutex> lock(mu);
    if (device < 0) return;
    if ((size_t)device >= seen.size()) seen.resize(device + 1, 0);
    if (seen[device]) return;
    seen[device] = 1;
    cudaFuncSetAttribute(sstc::k_oz_mm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sstc::kOzGemmSmem);
}

// exponents and digit slices of a dense operand (blocks kc * nrt + rt)
int slice_dense(ss_ctx *ctx, const OzOperand &op, Scratch &buf, unsigned char **sl, int **em) {
    const unsigned nrt = cdivu(op.rows, 128), nkc = cdivu(op.kdim, sstc::kOzK);
    OZ_ALLOC(ctx, buf.get(sl, (size_t)nrt * nkc * sstc::kOzStageA));
    OZ_ALLOC(ctx, buf.get(em, (size_t)op.rows));
    SS_CUDA_TRY(ctx, cudaMemsetAsync(*em, 0, sizeof(int) * op.rows, ctx->stream));
    const int64_t per_k = std::max<int64_t>(16, (int64_t)cdivu(op.kdim, std::max<unsigned>(1, 4 * ctx->sm_count / nrt)));
    ss_launch(ctx, SS_K_GEMM_TC, sstc::k_oz_expmax, dim3(nrt, cdivu(op.kdim, per_k)), 128, 0, ctx->stream, op, per_k,
              *em);
    const bool few = (int64_t)nrt * nkc <= 4ll * ctx->sm_count;
    ss_launch(ctx, SS_K_GEMM_TC, few ? sstc::k_oz_slice<512> : sstc::k_oz_slice<128>, dim3(nrt, nkc), few ? 512 : 128, 0,
              ctx->stream, op, (const int *)*em, *sl);
    return SS_OK;
}

int run_mm(ss_ctx *ctx, sstc::OzMM g, dim3 grid, int cls) {
    Scratch buf(ctx);
    OZ_ALLOC(ctx, buf.get(&g.status, 1));
    SS_CUDA_TRY(ctx, cudaMemsetAsync(g.status, 0, sizeof(int), ctx->stream));
    ss_launch(ctx, cls, sstc::k_oz_mm, grid, sstc::kOzThreads, sstc::kOzGemmSmem, ctx->stream, g);
    int h = 0;
    SS_CUDA_TRY(ctx, cudaMemcpyAsync(&h, g.status, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    SS_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
    if (h) return ctx->set_error(SS_ERR_TIMEOUT, "tensor-core product: a bounded wait ran out");
    SS_CUDA_TRY(ctx, cudaGetLastError());
    return SS_OK;
}

// dense product: mode 0 (G += alpha A B^T, split over the reduction) or mode 1
int dense_mm(ss_ctx *ctx, const OzOperand &A, const OzOperand &B, int mode, double alpha, double beta, double *out,
             int64_t ldo, double flops) {
    oz_attrs(ctx->device);
    Scratch buf(ctx);
    unsigned char *sa, *sb;
    int *ea, *eb;
    int rc;
    if ((rc = slice_dense(ctx, A, buf, &sa, &ea)) != SS_OK) return rc;
    if ((rc = slice_dense(ctx, B, buf, &sb, &eb)) != SS_OK) return rc;
    const int nrtA = (int)cdivu(A.rows, 128), nrtB = (int)cdivu(B.rows, 128), nkc = (int)cdivu(A.kdim, sstc::kOzK);
    const int nct = (int)cdivu(B.rows, 64);
    const int64_t tiles = (int64_t)nrtA * nct;
    int per = nkc;
    if (mode == 0) {
        // split the reduction until about two CTAs per SM
        const int64_t want = std::max<int64_t>(1, std::min<int64_t>(nkc, cdivu(2ll * ctx->sm_count, tiles)));
        per = (int)cdivu(nkc, want);
    }
    const int nsplit = (int)cdivu(nkc, per);
    sstc::OzMM g{};
    g.slA = sa; g.emA = ea; g.nrtA = nrtA; g.rowsA = A.rows;
    g.slB = sb; g.emB = eb; g.nrtB = nrtB; g.rowsB = B.rows;
    g.nkc = nkc; g.per = per; g.mode = mode; g.alpha = alpha; g.beta = beta;
    g.out = out; g.ldo = ldo;
    ctx->add_flops(SS_K_GEMM_TC, flops);
    ctx->add_tensor_flops(SS_K_GEMM_TC, kPieceTensorFlops * nrtA * nct * nkc);
    return run_mm(ctx, g, dim3(nct, nrtA, nsplit), SS_K_GEMM_TC);
}

// the lists of one analysis are freed apart: a failure to build one leaves the other, and the factors
// that use it, as they were
void free_plan(ss_symbolic *s) {
    OzPlan *pl = s->oz_plan;
    if (!pl) return;
    void *ptrs[] = {pl->d_tile_ptr, pl->d_pair_piece, pl->d_ent_ptr, pl->d_ent_e, pl->d_ent_off};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete pl;
    s->oz_plan = nullptr;
}

void free_samples(ss_symbolic *s) {
    OzSamples *sp = s->oz_samples;
    if (!sp) return;
    void *ptrs[] = {sp->d_rt, sp->d_ct, sp->d_ptr, sp->d_e, sp->d_t, sp->d_off};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete sp;
    s->oz_samples = nullptr;
}

// The lists are built on the host.  Where its memory does not do, the caller gets SS_ERR_OOM as for device
// memory: nothing may leave a C entry point, or a parallel region, as an exception.
// `bytes` of host lists are about to be allocated (ss_selftest_alloc_limit)
void host_room(const ss_ctx *ctx, size_t bytes) {
    if (ctx->alloc_limit >= 0 && bytes > (size_t)ctx->alloc_limit) throw std::bad_alloc();
}
template <typename F>
int guarded(ss_ctx *ctx, F &&build) {
    try {
        return build();
    } catch (const std::bad_alloc &) {
        return ctx->set_error(SS_ERR_OOM, "tensor-core product lists: host allocation failed");
    }
}
// body(row tile, counters) for every row tile in parallel, each thread with n counters of zero
template <typename T, typename F>
void each_row_tile(const ss_ctx *ctx, int32_t nrt, int64_t n, F &&body) {
    std::atomic<bool> failed{false};
#pragma omp parallel
    {
        std::vector<T> cnt;
        try {
            host_room(ctx, sizeof(T) * n);
            cnt.assign(n, 0);
        } catch (const std::bad_alloc &) {
            failed = true;
        }
#pragma omp for schedule(dynamic, 16)
        for (int32_t rt = 0; rt < nrt; ++rt) {
            if (failed || cnt.empty()) continue;
            try {
                body(rt, cnt);
            } catch (const std::bad_alloc &) {
                failed = true;
            }
        }
    }
    if (failed) throw std::bad_alloc();
}

// (tile, piece) pairs of the pattern -- for each 128-row tile the 32-column pieces that hold
// entries -- and the entries of every pair: CSR position (from the tile's first) and place in the
// pair's digit block
int plan_build(ss_symbolic *s) {
    ss_ctx *ctx = s->ctx;
    const int64_t n = s->n, npieces = (n + sstc::kOzK - 1) / sstc::kOzK;
    const int32_t nrt = (int32_t)cdivu(n, 128);
    std::vector<std::vector<int32_t>> pieces(nrt), counts(nrt);     // of a tile: pieces ascending, entries of each
    each_row_tile<int32_t>(ctx, nrt, npieces, [&](int32_t rt, std::vector<int32_t> &cnt) {
        const int64_t r1 = std::min<int64_t>(n, (rt + 1ll) * 128);
        std::vector<int32_t> &list = pieces[rt];
        for (int64_t p = s->rowptr[rt * 128ll]; p < s->rowptr[r1]; ++p)
            if (cnt[s->colind[p] / sstc::kOzK]++ == 0) list.push_back(s->colind[p] / sstc::kOzK);
        std::sort(list.begin(), list.end());
        for (int32_t pc : list) {
            counts[rt].push_back(cnt[pc]);
            cnt[pc] = 0;
        }
    });
    std::vector<int32_t> tile_ptr(nrt + 1, 0), pair_piece;
    std::vector<int64_t> ent_ptr(1, 0);
    for (int32_t rt = 0; rt < nrt; ++rt) {
        for (size_t u = 0; u < pieces[rt].size(); ++u) {
            pair_piece.push_back(pieces[rt][u]);
            ent_ptr.push_back(ent_ptr.back() + counts[rt][u]);
        }
        tile_ptr[rt + 1] = (int32_t)pair_piece.size();
    }
    std::vector<uint32_t> ent_e(std::max<int64_t>(1, s->nnz));
    std::vector<uint16_t> ent_off(std::max<int64_t>(1, s->nnz));
    each_row_tile<int64_t>(ctx, nrt, npieces, [&](int32_t rt, std::vector<int64_t> &at) {
        const int64_t r0 = rt * 128ll, r1 = std::min<int64_t>(n, r0 + 128), e0 = s->rowptr[r0];
        for (int32_t q = tile_ptr[rt]; q < tile_ptr[rt + 1]; ++q) at[pair_piece[q]] = ent_ptr[q];
        for (int64_t r = r0; r < r1; ++r)
            for (int64_t p = s->rowptr[r]; p < s->rowptr[r + 1]; ++p) {
                const int64_t o = at[s->colind[p] / sstc::kOzK]++;
                ent_e[o] = (uint32_t)(p - e0);
                ent_off[o] = (uint16_t)sstc::oz_offset((int)(r - r0), (int)(s->colind[p] % sstc::kOzK));
            }
    });
    OzPlan *pl = new OzPlan();
    pl->nrt = nrt;
    pl->npairs = (int64_t)pair_piece.size();
    s->oz_plan = pl;
    auto up = [&](auto **d, const auto &h) {
        cudaError_t e = ss_malloc(ctx, (void **)d, sizeof(h[0]) * std::max<size_t>(1, h.size()));
        if (e == cudaSuccess && !h.empty()) e = cudaMemcpy(*d, h.data(), sizeof(h[0]) * h.size(), cudaMemcpyHostToDevice);
        return e;
    };
    cudaError_t e = up(&pl->d_tile_ptr, tile_ptr);
    if (e == cudaSuccess) e = up(&pl->d_pair_piece, pair_piece);
    if (e == cudaSuccess) e = up(&pl->d_ent_ptr, ent_ptr);
    if (e == cudaSuccess) e = up(&pl->d_ent_e, ent_e);
    if (e == cudaSuccess) e = up(&pl->d_ent_off, ent_off);
    if (e != cudaSuccess) {
        cudaGetLastError();
        free_plan(s);
        return ctx->set_error(SS_ERR_OOM, "tensor-core product plan: device allocation failed");
    }
    return SS_OK;
}

int samples_count(ss_symbolic *s) {
    const int64_t n = s->n, nct = (n + 63) / 64;
    const int32_t nrt = (int32_t)cdivu(n, 128);
    std::vector<std::vector<int32_t>> cts(nrt), counts(nrt);
    each_row_tile<int32_t>(s->ctx, nrt, nct, [&](int32_t rt, std::vector<int32_t> &cnt) {
        const int64_t r0 = rt * 128ll, r1 = std::min<int64_t>(n, r0 + 128);
        for (int64_t r = r0; r < r1; ++r)
            for (int64_t p = s->rowptr[r]; p < s->rowptr[r + 1] && s->colind[p] <= r; ++p)
                if (cnt[s->colind[p] / 64]++ == 0) cts[rt].push_back(s->colind[p] / 64);
        std::sort(cts[rt].begin(), cts[rt].end());
        for (int32_t ct : cts[rt]) {
            counts[rt].push_back(cnt[ct]);
            cnt[ct] = 0;
        }
    });
    std::unique_ptr<OzSamples> sp(new OzSamples());
    sp->ptr.assign(1, 0);
    sp->first.assign(nrt, 0);
    for (int32_t rt = 0; rt < nrt; ++rt) {
        sp->first[rt] = (int64_t)sp->rts.size();
        for (size_t u = 0; u < cts[rt].size(); ++u) {
            sp->rts.push_back(rt);
            sp->cts.push_back(cts[rt][u]);
            sp->ptr.push_back(sp->ptr.back() + counts[rt][u]);
        }
    }
    sp->ntiles = (int64_t)sp->rts.size();
    s->oz_samples = sp.release();
    return SS_OK;
}

int samples_build(ss_symbolic *s) {
    ss_ctx *ctx = s->ctx;
    OzSamples *sp = s->oz_samples;
    const int64_t n = s->n, nct = (n + 63) / 64;
    const int32_t nrt = (int32_t)cdivu(n, 128);
    const size_t m = (size_t)std::max<int64_t>(1, sp->ptr.back());
    std::vector<uint32_t> e(m), t(m);
    std::vector<uint16_t> off(m);
    each_row_tile<int64_t>(ctx, nrt, nct, [&](int32_t rt, std::vector<int64_t> &at) {
        const int64_t r0 = rt * 128ll, r1 = std::min<int64_t>(n, r0 + 128);
        const int64_t t1 = rt + 1 < nrt ? sp->first[rt + 1] : sp->ntiles;
        for (int64_t u = sp->first[rt]; u < t1; ++u) at[sp->cts[u]] = sp->ptr[u];
        for (int64_t r = r0; r < r1; ++r)
            for (int64_t p = s->rowptr[r]; p < s->rowptr[r + 1] && s->colind[p] <= r; ++p) {
                const int64_t c = s->colind[p], o = at[c / 64]++;
                const int32_t *b = s->colind.data() + s->rowptr[c], *z = s->colind.data() + s->rowptr[c + 1];
                e[o] = (uint32_t)p;
                t[o] = (uint32_t)(std::lower_bound(b, z, (int32_t)r) - s->colind.data());   // (c, r): the pattern is symmetric
                off[o] = (uint16_t)((r - r0) * 64 + c % 64);
            }
    });
    auto up = [&](auto **d, const auto &h) {
        cudaError_t er = ss_malloc(ctx, (void **)d, sizeof(h[0]) * std::max<size_t>(1, h.size()));
        if (er == cudaSuccess && !h.empty()) er = cudaMemcpy(*d, h.data(), sizeof(h[0]) * h.size(), cudaMemcpyHostToDevice);
        return er;
    };
    cudaError_t er = up(&sp->d_rt, sp->rts);
    if (er == cudaSuccess) er = up(&sp->d_ct, sp->cts);
    if (er == cudaSuccess) er = up(&sp->d_ptr, sp->ptr);
    if (er == cudaSuccess) er = up(&sp->d_e, e);
    if (er == cudaSuccess) er = up(&sp->d_t, t);
    if (er == cudaSuccess) er = up(&sp->d_off, off);
    if (er != cudaSuccess) {
        cudaGetLastError();
        free_samples(s);
        return ctx->set_error(SS_ERR_OOM, "sampled product plan: device allocation failed");
    }
    sp->rts.clear(), sp->rts.shrink_to_fit();
    sp->cts.clear(), sp->cts.shrink_to_fit();
    sp->ptr.clear(), sp->ptr.shrink_to_fit();
    sp->first.clear(), sp->first.shrink_to_fit();
    return SS_OK;
}

// row exponents of one value array on the pattern, into v (device memory from buf, or owned by v
// when buf is null)
int vals_make(ss_symbolic *s, const double *vals, OzVals *v, Scratch *buf) {
    ss_ctx *ctx = s->ctx;
    v->vals = vals;
    if (buf) {
        OZ_ALLOC(ctx, buf->get(&v->em, (size_t)s->n));
    } else {
        OZ_ALLOC(ctx, ss_malloc(ctx, (void **)&v->em, sizeof(int) * s->n));
    }
    oz_attrs(ctx->device);
    ss_launch(ctx, SS_K_SPMM_TC, sstc::k_oz_csr_expmax, cdivu(s->n * 32, 256), 256, 0, ctx->stream, s->n,
              (const int64_t *)s->d_rowptr, vals, v->em);
    SS_CUDA_TRY(ctx, cudaGetLastError());
    return SS_OK;
}

// row exponents of value array `which` (0: A, 1: B) of f, made on first use
int vals_get(ss_numeric *f, int which, OzVals **out) {
    *out = f->oz[which];
    if (*out) return SS_OK;
    OzVals *v = new (std::nothrow) OzVals();
    if (!v) return f->sym->ctx->set_error(SS_ERR_OOM, "tensor-core product: host allocation failed");
    const int rc = vals_make(f->sym, which == 0 ? f->a_vals : f->b_vals, v, nullptr);
    if (rc != SS_OK) {
        delete v;
        return rc;
    }
    f->oz[which] = *out = v;   // freed with the factor
    return SS_OK;
}

// pass p adds alpha[p] diag(colscale[p]) M_p X, M_p the array of v[p]; the first
// pass overwrites Y
int spmm_core(ss_symbolic *s, int npass, OzVals *const *v, const double *const *colscale, const double *alpha,
              const double *X, int64_t ldx, int k, double *Y, int64_t ldy) {
    ss_ctx *ctx = s->ctx;
    int rc;
    if (!s->oz_plan && (rc = guarded(ctx, [&] { return plan_build(s); })) != SS_OK) return rc;
    Scratch buf(ctx);
    unsigned char *sx;
    int *ex;
    // operand rows of X = its k columns, reduction over the n rows
    const OzOperand xo{X, 1, ldx, k, s->n};
    if ((rc = slice_dense(ctx, xo, buf, &sx, &ex)) != SS_OK) return rc;
    const OzPlan *pl = s->oz_plan;
    for (int p = 0; p < npass; ++p) {
        sstc::OzMM g{};
        g.emA = v[p]->em; g.nrtA = pl->nrt; g.rowsA = s->n;
        g.tile_ptr = pl->d_tile_ptr; g.pair_piece = pl->d_pair_piece;
        g.ent_ptr = pl->d_ent_ptr; g.ent_e = pl->d_ent_e; g.ent_off = pl->d_ent_off;
        g.rowptr = s->d_rowptr; g.vals = v[p]->vals;
        g.slB = sx; g.emB = ex; g.nrtB = (int)cdivu(k, 128); g.rowsB = k;
        g.mode = 1; g.alpha = alpha[p]; g.beta = p == 0 ? 0.0 : 1.0; g.colscale = colscale[p];
        g.out = Y; g.ldo = ldy;
        ctx->add_flops(SS_K_SPMM_TC, 2.0 * (double)s->nnz * k);
        ctx->add_tensor_flops(SS_K_SPMM_TC, kPieceTensorFlops * (double)pl->npairs * cdivu(k, 64));
        if ((rc = run_mm(ctx, g, dim3(cdivu(k, 64), pl->nrt, 1), SS_K_SPMM_TC)) != SS_OK) return rc;
    }
    return SS_OK;
}

}  // namespace

bool oz_dense_ok(const ss_ctx *ctx, int64_t n, int k1, int k2) {
    return ctx->gemm_mode == SS_GEMM_TENSOR && n >= 2048 && k1 >= 48 && k2 >= 48;
}

bool oz_spmm_ok(const ss_numeric *f, int k) {
    return f->sym->ctx->gemm_mode == SS_GEMM_TENSOR && f->sym->n >= 2048 && k >= 48 && !f->oz_failed;
}

int oz_gram(ss_ctx *ctx, const double *X, int64_t ldx, int64_t n, int k1, const double *Y, int64_t ldy, int k2,
            double *G) {
    // operand rows = the columns of X and of Y, reduction over the n rows; G zeroed here
    SS_CUDA_TRY(ctx, cudaMemsetAsync(G, 0, sizeof(double) * k1 * k2, ctx->stream));
    const OzOperand a{X, 1, ldx, k1, n}, b{Y, 1, ldy, k2, n};
    return dense_mm(ctx, a, b, 0, 1.0, 0.0, G, k2, 2.0 * (double)n * k1 * k2);
}

int oz_gemm(ss_ctx *ctx, const double *X, int64_t ldx, int64_t n, int k1, const double *Q, int k2, int transq,
            double alpha, double beta, double *Y, int64_t ldy) {
    // operand rows = the rows of X and the columns of the effective k1 x k2 Q, reduction over k1
    const OzOperand a{X, ldx, 1, n, k1};
    const OzOperand b = transq ? OzOperand{Q, k1, 1, k2, k1} : OzOperand{Q, 1, k2, k2, k1};
    return dense_mm(ctx, a, b, 1, alpha, beta, Y, ldy, 2.0 * (double)n * k1 * k2);
}

int oz_spmm(ss_numeric *f, int npass, const int *which, const double *const *colscale, const double *alpha,
            const double *X, int64_t ldx, int k, double *Y, int64_t ldy) {
    int rc;
    OzVals *v[2] = {nullptr, nullptr};
    for (int p = 0; p < npass; ++p)
        if ((rc = vals_get(f, which[p], &v[p])) != SS_OK) return rc;
    return spmm_core(f->sym, npass, v, colscale, alpha, X, ldx, k, Y, ldy);
}

int oz_spmm_vals(ss_symbolic *s, const double *a, const double *b, const double *alpha, const double *beta,
                 const double *X, int64_t ldx, int k, double *Y, int64_t ldy) {
    Scratch buf(s->ctx);
    OzVals va, vb;
    int rc;
    if ((rc = vals_make(s, a, &va, &buf)) != SS_OK) return rc;
    if (beta && (rc = vals_make(s, b, &vb, &buf)) != SS_OK) return rc;
    OzVals *v[2] = {&va, &vb};
    const double *cs[2] = {alpha, beta};
    const double al[2] = {1.0, 1.0};
    return spmm_core(s, beta ? 2 : 1, v, cs, al, X, ldx, k, Y, ldy);
}

// Y = diag(alpha) A X + diag(beta) B X on the tensor cores when the mode, the sizes and the
// value arrays (the factor's own A and B) allow, else on the CUDA cores
int spmm_f(ss_numeric *f, const double *a, const double *b, const double *alpha, const double *beta, const double *X,
           int64_t ldx, int k, double *Y, int64_t ldy) {
    ss_symbolic *s = f->sym;
    const int ia = a == f->a_vals ? 0 : (a == f->b_vals ? 1 : -1);
    const int ib = !beta ? 0 : (b == f->a_vals ? 0 : (b == f->b_vals ? 1 : -1));
    if (oz_spmm_ok(f, k) && ia >= 0 && ib >= 0) {
        const int which[2] = {ia, ib};
        const double *cs[2] = {alpha, beta};
        const double al[2] = {1.0, 1.0};
        const int rc = oz_spmm(f, beta ? 2 : 1, which, cs, al, X, ldx, k, Y, ldy);
        if (rc != SS_ERR_OOM) return rc;
        // the plan or the digits of X do not fit beside the factor: CUDA cores from now on
        f->oz_failed = true;
        s->ctx->err.clear();
    }
    return spmm_launch_ld(s, a, b, alpha, beta, X, ldx, k, Y, ldy);
}

void oz_free_numeric(ss_numeric *f) {
    auto drop = [](OzVals *&v) {
        if (!v) return;
        if (v->em) cudaFree(v->em);
        delete v;
        v = nullptr;
    };
    for (OzVals *&v : f->oz) drop(v);
}

// Whether X Y^T sampled on the pattern runs on the tensor cores: 32-bit CSR positions, enough columns to
// fill a piece, and the quicker of two estimates in picoseconds.  CUDA cores: two multiply-adds an entry
// and column and the sums over the lanes, worth 300 columns.  Tensor cores: the launches, every 128 x 64
// tile that holds an entry in full, and the digits of X and X diag(lambda).  Measured / estimated, us,
// CUDA cores and tensor cores: N = 20,000, 17 entries a row in 469 tiles, ne = 48 368 / 366 and 286 / 283,
// ne = 1,640 2,269 / 2,045 and 1,479 / 1,443; 9 a row 209 / 194 and 281 / 283; N = 8,000, 9 scattered
// entries a row in 4,031 tiles 99 / 78 and 1,136 / 1,281; N = 16,384, 472 a row, ne = 1,640 50,700 and 6,540.
bool oz_sddmm_ok(ss_symbolic *s, int ne) {
    if (s->ctx->gemm_mode != SS_GEMM_TENSOR || s->n < 2048 || ne < 48 || s->nnz >= (1ll << 32)) return false;
    const double cuda = 3.1 * (double)s->nnz * (ne + 300.0), rest = 1.3e8 + 20.0 * (double)s->n * ne;
    if (cuda <= rest) return false;
    if (!s->oz_samples && guarded(s->ctx, [&] { return samples_count(s); }) != SS_OK) {
        s->ctx->err.clear();                   // CUDA cores
        return false;
    }
    return cuda > rest + (double)s->oz_samples->ntiles * (2.5e5 + 700.0 * ne);
}

int oz_sddmm(ss_symbolic *s, const double *X, const double *lambda, int ne, double *grad_a, double *grad_b) {
    ss_ctx *ctx = s->ctx;
    int rc;
    if (!s->oz_samples->d_rt && (rc = guarded(ctx, [&] { return samples_build(s); })) != SS_OK) return rc;
    const OzSamples *sp = s->oz_samples;
    oz_attrs(ctx->device);
    Scratch buf(ctx);
    unsigned char *sx, *sl;
    int *ex, *el;
    // operand rows = rows of X (and of X diag(lambda)), reduction over the ne columns
    OzOperand x{X, ne, 1, s->n, ne};
    if ((rc = slice_dense(ctx, x, buf, &sx, &ex)) != SS_OK) return rc;
    const int nkc = (int)cdivu(ne, sstc::kOzK), nrt = (int)cdivu(s->n, 128);
    for (int pass = 0; pass < 2; ++pass) {
        double *out = pass == 0 ? grad_a : grad_b;
        if (!out || sp->ntiles == 0) continue;
        sstc::OzMM g{};
        g.slA = sx; g.emA = ex; g.nrtA = nrt; g.rowsA = s->n;
        g.slB = sx; g.emB = ex; g.nrtB = nrt; g.rowsB = s->n;
        if (pass == 1) {
            x.kscale = lambda;
            if ((rc = slice_dense(ctx, x, buf, &sl, &el)) != SS_OK) return rc;
            g.slB = sl; g.emB = el;
        }
        g.nkc = nkc; g.per = nkc; g.mode = 2; g.alpha = pass == 0 ? 1.0 : -1.0; g.out = out;
        g.samp_rt = sp->d_rt; g.samp_ct = sp->d_ct; g.samp_ptr = sp->d_ptr;
        g.samp_e = sp->d_e; g.samp_t = sp->d_t; g.samp_off = sp->d_off;
        ctx->add_tensor_flops(SS_K_SDDMM, kPieceTensorFlops * (double)sp->ntiles * nkc);
        if ((rc = run_mm(ctx, g, dim3((unsigned)sp->ntiles, 1, 1), SS_K_SDDMM)) != SS_OK) return rc;
    }
    return SS_OK;
}

void oz_free_symbolic(ss_symbolic *s) {
    free_samples(s);
    free_plan(s);
}
