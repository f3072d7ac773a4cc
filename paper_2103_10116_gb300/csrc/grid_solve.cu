// grid_solve.cu -- host side of the one-launch solves over the device
// (grid_solve.cuh): partition, workspace, launch, result.
#include "grid_solve.cuh"

#include <algorithm>
#include <atomic>

namespace spx {

template <class T, class V, bool PRE, bool COMPACT>
int grid_launch(spx_ctx *ctx, const GridArgs &A, int solver, int blocks, int threads, int r);
#define SPX_GRID(T, V)                                                                                \
    extern template int grid_launch<T, V, false, false>(spx_ctx *, const GridArgs &, int, int, int, int); \
    extern template int grid_launch<T, V, true, false>(spx_ctx *, const GridArgs &, int, int, int, int);  \
    extern template int grid_launch<T, V, false, true>(spx_ctx *, const GridArgs &, int, int, int, int);  \
    extern template int grid_launch<T, V, true, true>(spx_ctx *, const GridArgs &, int, int, int, int);
SPX_GRID(double, double)
SPX_GRID(float, float)
SPX_GRID(double, float)
#undef SPX_GRID

namespace {

// Rows per block from which a further block is taken.  Fewer blocks make each sum
// cheaper (grid_solve.cuh), more blocks share the FP64 work: FP64 BiCGSTAB on 12 000
// rows of 20 random columns 0.77 ms at 128, 0.90 at 256, 1.25 at 512; mixed CG on 8100
// 5-point rows 1.51 / 1.40 / 1.42 ms, mixed BiCGSTAB on 30 001 random rows 0.64 / 0.63
// / 0.72 ms.
constexpr int kGridMinRows64 = 128;
constexpr int kGridMinRows32 = 256;
// Systems from which this route is faster than one cluster (CG in one precision,
// cluster.cu) or one SM (the others, the batched kernel as a batch of one), measured
// in ms, the other route first.  CG FP64: 8100 rows 1.36 / 2.05, 15 625 rows 0.86 / 0.88;
// 27-point 10 648 rows, whose slices do not fit one cluster, 1.10 / 0.55; FP32: 8100 rows
// 0.14 / 0.27.  Against one SM what counts is the entries: mixed CG on 1296 5-point rows (6336
// entries) 0.44 / 0.50, 1600 rows (7840) 0.56 / 0.57, 1764 rows (8652) 0.71 / 0.55, 1331 27-point rows
// (29 791) 0.65 / 0.21; mixed BiCGSTAB 1000 7-point rows (6400) 0.24 / 0.26, 1331 rows (8591) 0.36 / 0.25;
// FP64 729 rows (4617) 0.34 / 0.35, 1000 rows 0.40 / 0.38; 256 rows of 20 0.25 / 0.32, 520 rows 0.49 / 0.38,
// those with grids for one SM 0.46 / 0.55, 1000 rows 1.01 / 0.85.  ELL and COO
// have the general path otherwise, slower at every size: CG FP64 on 1600 5-point rows in ELL
// 3.7 / 0.93, mixed CG on 8100 rows in COO 8.5 / 1.4, CGS on 97 336 7-point rows in ELL 3.6 / 1.9.
// So has Jacobi: CG FP64 on 400 5-point rows 2.0 / 0.52, on 262 144 7-point rows 6.9 / 4.0, mixed
// on 4096 5-point rows 5.8 / 1.5; BiCGSTAB FP64 on 300 random rows 0.90 / 0.16, on 30 000 in COO
// 0.65 / 0.25.
constexpr int64_t kGridCgRows64 = 14336;
constexpr int64_t kGridCgRows32 = 16385;
constexpr int64_t kGridCgRowsOff = 4096;  // ... where the cluster does not keep the matrix on chip
constexpr int64_t kGridRows = 512;
constexpr int64_t kGridEntries32 = 8192;  // FP32 products (mixed precision among them)
constexpr int64_t kGridEntries64 = 5632, kGridEntries64Sm = 9216;  // FP64: the first plus the second over the SMs
constexpr size_t kGridWordBytes = grid_words(kGridMaxBlocks) * 8;

// Solves of this route that are running on each device: with others at its side, a solve takes the
// COMPACT kernel, which leaves room on the SMs for a second one (its results are the same bits).
// A cooperative launch waits until all its blocks fit, so without it solves of several contexts
// ran one after the other.  us per solve, 16 contexts at once, without / with, and alone without /
// with: CG mixed 46^3 1304 / 778, 1402 / 1507; 63^3 2137 / 1273, 2161 / 2265; FP64 40^3 1604 /
// 996, 1617 / 1654; BiCGSTAB FP64 35^3 1781 / 775, 1872 / 1830.  Rows of 12 or more entries keep
// the FP64 pipe or the gathers busy as they are (BiCGSTAB mixed, 30 001 rows of 20: 373 / 577).
std::atomic<int> g_grid_running[256];
constexpr double kGridCompactMeanLen = 12.0;

struct Running {
    std::atomic<int> *n;
    bool others;
    explicit Running(int dev) : n(dev >= 0 && dev < 256 ? &g_grid_running[dev] : nullptr)
    {
        others = n && n->fetch_add(1) > 0;
    }
    ~Running()
    {
        if (n) n->fetch_sub(1);
    }
};

template <class T, class V>
int launch(spx_ctx *ctx, const GridArgs &g, bool jacobi, bool compact, int solver, int blocks, int threads, int r)
{
    if (compact)
        return jacobi ? grid_launch<T, V, true, true>(ctx, g, solver, blocks, threads, r)
                      : grid_launch<T, V, false, true>(ctx, g, solver, blocks, threads, r);
    return jacobi ? grid_launch<T, V, true, false>(ctx, g, solver, blocks, threads, r)
                  : grid_launch<T, V, false, false>(ctx, g, solver, blocks, threads, r);
}

// The record of a launch on the context's stream; an error unless block 0 finished and no block reported any.
int grid_result(spx_ctx *ctx, const GridOut *out, GridOut &h)
{
    SPX_CUDA(cudaMemcpyAsync(&h, out, sizeof(h), cudaMemcpyDeviceToHost, ctx->stream));
    SPX_CUDA(cudaStreamSynchronize(ctx->stream));
    if (h.done && !h.err) return SPX_OK;
    return check_dev_err(ctx) != SPX_OK ? SPX_ERR_TIMEOUT : fail(SPX_ERR_CUDA, "the solve did not finish");
}

// Block 0 reports a result while block 1 waits, for a millisecond, for a sum that block 0 has no part in.
__global__ void k_grid_selftest(GridArgs A)
{
    __shared__ double buf[2 * kGridBlockMax], total[4];
    __shared__ int s_dead;
    GridTeam tm;
    tm.words = A.words;
    tm.buf = buf;
    tm.total = total;
    tm.s_dead = &s_dead;
    tm.limit = 2000000;
    if (threadIdx.x == 0) s_dead = 0;
    __syncthreads();
    float v = 1.f;
    const bool ok = blockIdx.x == 0 || tm.sum(v);
    if (threadIdx.x != 0) return;
    if (!ok) grid_error(A, DEVERR_QUEUE_TIMEOUT);
    if (blockIdx.x == 0) grid_report(A, GridOut{1, SPX_CONVERGED, 0, 0u, 0, 0.0, 0.0});
}

}  // namespace

// See spx_internal.cuh.
int grid_selftest(spx_ctx *ctx)
{
    const size_t words = grid_words(2) * 8;
    DBuf w;
    SPX_TRY(dbuf_alloc(ctx, w, words + sizeof(GridOut)));
    GridArgs g = {};
    g.words = w.as<unsigned long long>();
    g.out = reinterpret_cast<GridOut *>(w.as<char>() + words);
    g.err = ctx->dev_err;
    cudaError_t e = cudaMemsetAsync(w.p, 0, words + sizeof(GridOut), ctx->stream);
    if (e == cudaSuccess) {
        k_grid_selftest<<<2, 32, 0, ctx->stream>>>(g);
        e = cudaGetLastError();
    }
    GridOut h;
    const int st = e == cudaSuccess ? grid_result(ctx, g.out, h) : cuda_fail(e, "k_grid_selftest");
    dbuf_free(ctx, w);
    return st;
}

// See spx_internal.cuh.
int grid_solve(spx_ctx *ctx, spx_matrix *A, const void *b, void *x, int solver, double tol, int64_t maxit,
               int precision, bool jacobi, spx_solve_info *info)
{
    if (A->n < 1 || A->nnz < 1) return SPX_ERR_UNSUPPORTED;
    const bool csr = A->format == SPX_CSR && A->rp.p;
    const bool ell = A->ell_w > 0 && (A->format == SPX_ELL || (A->format == SPX_HYB && A->coo_nnz == 0));
    const bool coo = A->format == SPX_COO && A->coo_nnz > 0;
    if (!csr && !ell && !coo) return SPX_ERR_UNSUPPORTED;
    if (solver != SPX_CG && solver != SPX_BICGSTAB && solver != SPX_CGS) return SPX_ERR_UNSUPPORTED;
    const bool mixed = precision == SPX_PREC_MIXED;
    const DBuf &val = csr ? A->val : ell ? A->ell_val : A->coo_val;
    const DBuf &val32 = csr ? A->val32 : ell ? A->ell_val32 : A->coo_val32;
    if (mixed ? A->dtype != SPX_F64 || !val32.p : (precision == SPX_PREC_F64 ? SPX_F64 : SPX_F32) != A->dtype)
        return SPX_ERR_UNSUPPORTED;  // the general path reports the mismatch
    // one thread per row: rows of similar length only (the row-block SpMV's rule)
    if ((double)A->max_len > 2.0 * A->mean_len + 8.0) return SPX_ERR_UNSUPPORTED;
    const int64_t sms = std::min<int64_t>(ctx->grid_sms, kGridMaxBlocks);
    const int64_t from = !csr || jacobi                ? 1  // the small routes take plain CSR only
                         : solver != SPX_CG || mixed   ? kGridRows
                         : !cluster_cg_on_chip(ctx, A) ? kGridCgRowsOff
                         : precision == SPX_PREC_F64   ? kGridCgRows64
                                                       : kGridCgRows32;
    if (A->n < from) return SPX_ERR_UNSUPPORTED;
    const int64_t entries = precision == SPX_PREC_F64 ? kGridEntries64 + kGridEntries64Sm / sms : kGridEntries32;
    if (from == kGridRows && A->nnz < entries) return SPX_ERR_UNSUPPORTED;
    const int64_t min_rows = precision == SPX_PREC_F64 ? kGridMinRows64 : kGridMinRows32;
    const int64_t want = std::min<int64_t>(sms, ceil_div(A->n, min_rows));
    const int64_t rows = (int64_t)round_up((size_t)ceil_div(A->n, want), 32);
    if (rows > 4 * kGridBlockMax) return SPX_ERR_UNSUPPORTED;
    const int r = rows <= kGridBlockMax ? 1 : rows <= 2 * kGridBlockMax ? 2 : 4;
    const int threads = (int)round_up((size_t)ceil_div(rows, (int64_t)r), 32);
    const int blocks = (int)ceil_div(A->n, rows);
    const int64_t cap = ell ? A->ell_w * rows : std::min<int64_t>(A->max_len * rows, A->nnz);
    const size_t smem = A->dtype == SPX_F64 && !mixed ? grid_smem<double>((int)std::min<int64_t>(cap, 1 << 20))
                                                      : grid_smem<float>((int)std::min<int64_t>(cap, 1 << 20));
    if (smem > (size_t)ctx->max_smem_optin - 1024) return SPX_ERR_UNSUPPORTED;
    // workspace: slots and result | gathered vector | gathered FP64 x
    const size_t head = kGridWordBytes + 256, vec = round_up((size_t)A->n * 8, 256);
    if (!A->grid_work.p) SPX_TRY(dbuf_alloc(ctx, A->grid_work, head + 2 * vec));  // stream-ordered with its use
    char *w = A->grid_work.as<char>();
    GridArgs g;
    g.n = (int)A->n;
    g.rows = (int)rows;
    g.cap = (int)cap;
    g.rp = csr ? A->rp.as<int>() : nullptr;
    g.crow = coo ? A->coo_row.as<int>() : nullptr;
    g.nnz = (int)A->nnz;
    g.ell_ld = ell ? A->ell_ld : 0;
    g.ell_w = (int)A->ell_w;
    g.col = csr ? A->col.as<int>() : ell ? A->ell_col.as<int>() : A->coo_col.as<int>();
    g.val = mixed ? val32.p : val.p;
    g.val64 = val.p;
    g.b = b;
    g.x = x;
    g.ps = w + head;
    g.xs = reinterpret_cast<double *>(w + head + vec);
    g.words = reinterpret_cast<unsigned long long *>(w);
    g.out = reinterpret_cast<GridOut *>(w + kGridWordBytes);
    g.err = ctx->dev_err;
    g.tol = tol;
    g.maxit = (long long)maxit;
    SPX_CUDA(cudaMemsetAsync(w, 0, grid_words(blocks) * 8, ctx->stream));
    SPX_CUDA(cudaMemsetAsync(g.out, 0, sizeof(GridOut), ctx->stream));
    const Running running(ctx->device);
    const bool f64 = A->dtype == SPX_F64 && !mixed;
    const bool compact = running.others && A->mean_len < kGridCompactMeanLen && !(f64 && r == 4);
    const int st = mixed ? launch<double, float>(ctx, g, jacobi, compact, solver, blocks, threads, r)
                   : f64 ? launch<double, double>(ctx, g, jacobi, compact, solver, blocks, threads, r)
                         : launch<float, float>(ctx, g, jacobi, compact, solver, blocks, threads, r);
    if (st != SPX_OK) return st;
    GridOut h;
    SPX_TRY(grid_result(ctx, g.out, h));
    info->status = h.status;
    info->iterations = h.iters;
    info->restarts = h.restarts;
    info->relres_recurrence = h.relres;
    info->relres_true = h.relres_true;
    if (mixed) info->inner_iterations = h.iters;
    return SPX_OK;
}

}  // namespace spx
