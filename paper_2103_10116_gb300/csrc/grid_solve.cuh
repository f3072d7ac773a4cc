// grid_solve.cuh -- a whole Krylov solve in one cooperative launch over the
// device: CG, BiCGSTAB and CGS (FP64 or FP32), mixed-precision CG with reliable
// updates, and FP64 refinement around FP32 BiCGSTAB / CGS, for systems (CSR, ELL, COO) of
// rows of similar length whose matrix fits the SMs' shared memory together; without
// preconditioner or with Jacobi (mixed CG then as refinement around FP32 CG).
//
// The general path pays three to five launches and as many device-wide
// reductions per iteration, 15 to 25 us however small the system (FP32 CG on a
// 7-point stencil of 97 336 rows: 19 us per iteration for 1 us of HBM traffic;
// here 7.0 us, its mixed solve to 1e-8 3.05 -> 1.11 ms; FP64 BiCGSTAB on 30 001
// rows of 20 random columns 45 -> 25 us per iteration).
// Here block k owns rows [k S, (k+1) S): it copies its slice of the column
// indices and values into shared memory once, keeps its slices of the solver's
// vectors in registers (R rows per thread), and only the vector that a product
// gathers from passes through global memory (L2).  A dot product is a block sum
// published in a slot of its block; every block reads all slots and adds them in
// block order, so the sum is also the grid barrier, every block holds the same
// bits and takes the same decisions, and the result does not depend on timing.
// What bounds an iteration is then the latency of its barriers and gathers and,
// in FP64, the SMs' FP64 rate.
//
// The launch is cooperative (all blocks resident), so every wait ends; each
// wait is bounded all the same: a block whose wait gives up leaves the kernel, setting
// the context's error word and the result record's, as do the others when their waits
// run out; those may have finished, so the host takes a result only from a record
// without errors.
#pragma once

#include "dev_common.cuh"
#include "spx_internal.cuh"

namespace spx {

constexpr int kGridBlockMax = 512;   // threads per block
constexpr int kGridMaxBlocks = 160;  // blocks: five slots per lane of the warp that reads them
constexpr int kGridWords = 4;        // words per slot: two sums, two words each
constexpr int kGridCopies = 16;      // places a block writes its slot to
constexpr int kGridRestarts = 3;
constexpr float kGridRuDelta2 = 0.01f;  // reliable updates: delta^2, delta = 0.1 (as run_cg_reliable)

constexpr long long kGridWaitCycles = 2000000000LL;  // a wait's limit, about a second

// Result record, zero at launch: block 0 writes all but err, done = 1 among it; err: any
// block's errors, and those that the context's word held already.
struct GridOut {
    int done, status, restarts;
    unsigned err;
    long long iters;
    double relres, relres_true;
};

struct GridArgs {
    int n, rows, cap;  // rows of the system and per block, entries the shared slice holds
    const int *rp, *col;  // CSR; COO: crow instead of rp (rows found by search), nnz
    const int *crow;
    int nnz;
    int64_t ell_ld;  // ELL (col, val column-major; rp, crow null): rows between slabs
    int ell_w;
    const void *val, *val64;  // the values the products use; the FP64 values of a mixed solve
    const void *b;
    void *x;
    void *ps;  // the gathered vector
    double *xs;  // mixed: the gathered FP64 x
    unsigned long long *words;  // grid_words(blocks), zero at launch
    GridOut *out;
    unsigned *err;
    double tol;
    long long maxit;
};

// The blocks of the grid: sums over all of them.
//
// Two forms, by what the sum has to order.  Both end with every block adding all
// blocks' values in block order.  Measured with 152 blocks (clocks per sum, FP64
// arithmetic apart; a store takes about 2000 clocks to be seen from the other die):
//   * sums that publish no memory (p.q, r.r, ...) carry their data in words tagged
//     with the sum's number, which every block polls directly: 3250, and 2250 with 32
//     blocks.  A block writes its slot to kGridCopies places and polls the place of
//     its group of blocks: all blocks polling one place took 5500;
//   * sums and barriers that publish a vector count arrivals on one word, between
//     fences, then read plain slots: 4100 (2700 without slots), against 5500 to 7200
//     for tagged words with the same fences, whose polling slows the fences.
struct GridTeam {
    unsigned long long *words;
    double *buf;    // shared: 2 kGridBlockMax
    double *total;  // shared: 4
    int *s_dead;    // shared: a wait gave up
    long long limit = kGridWaitCycles;
    unsigned epoch = 0, fenced = 0;

    static __device__ __forceinline__ void put(unsigned long long *slot, unsigned long long a, unsigned long long b)
    {
        asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(slot), "l"(a), "l"(b) : "memory");
    }
    static __device__ __forceinline__ void get(const unsigned long long *slot, unsigned long long &a,
                                               unsigned long long &b)
    {
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(slot) : "memory");
    }
    static __device__ __forceinline__ void fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

    __device__ __forceinline__ void give_up() { *s_dead = 1; }

    // s[q] (valid in warp 0's lanes) = the value of block l + 32 k in a[q][k], all blocks' values
    // ready.  Tagged words: a slot is rewritten two sums later, by when every block has
    // published the sum between and so has read this one; each word carries the sum's number
    // in its upper half, so a slot is read whole or not at all.  The values read before the
    // sum feed it, so a vector those reads gathered from may be rewritten after it.
    template <class T, int NV> __device__ __forceinline__ void all_tagged(const T *s, T (*a)[kGridMaxBlocks / 32], int l)
    {
        constexpr int NS = kGridMaxBlocks / 32;
        const int nb = gridDim.x;
        const size_t place = (size_t)nb * kGridWords;
        unsigned long long *set = words + (epoch & 1u) * kGridCopies * place;
        const unsigned long long tag = (unsigned long long)epoch << 32;
        if (l < kGridCopies) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                unsigned long long bits;
                if constexpr (sizeof(T) == 8) bits = (unsigned long long)__double_as_longlong((double)s[q]);
                else bits = (unsigned long long)__float_as_uint((float)s[q]);
                put(set + l * place + (size_t)blockIdx.x * kGridWords + 2 * q, tag | (bits & 0xffffffffull),
                    tag | (bits >> 32));
            }
        }
        const unsigned long long *mine = set + (size_t)(blockIdx.x * kGridCopies / nb) * place;
        unsigned long long w0[NV][NS], w1[NV][NS];
        const long long t0 = clock64();
        bool ready;
        do {
            ready = true;
#pragma unroll
            for (int q = 0; q < NV; ++q)
#pragma unroll
                for (int k = 0; k < NS; ++k) {
                    w0[q][k] = w1[q][k] = tag;  // a block past the last one: 0
                    if (l + 32 * k < nb) get(mine + (size_t)(l + 32 * k) * kGridWords + 2 * q, w0[q][k], w1[q][k]);
                }
#pragma unroll
            for (int q = 0; q < NV; ++q)
#pragma unroll
                for (int k = 0; k < NS; ++k)
                    ready = ready && (unsigned)(w0[q][k] >> 32) == epoch && (unsigned)(w1[q][k] >> 32) == epoch;
            if (!ready && clock64() - t0 > limit) {
                give_up();
                break;
            }
        } while (!ready);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NV; ++q)
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                const unsigned long long bits = (w0[q][k] & 0xffffffffull) | (w1[q][k] << 32);
                if constexpr (sizeof(T) == 8) a[q][k] = (T)__longlong_as_double((long long)bits);
                else a[q][k] = (T)__uint_as_float((unsigned)bits);
            }
    }

    // The same with release / acquire: what the grid's threads wrote before the call is
    // visible after it.  Slots alternate between two sets; a block writes a set again only
    // past the fenced barrier between, at which every block has read this one.
    template <class T, int NV> __device__ __forceinline__ void all_fenced(const T *s, T (*a)[kGridMaxBlocks / 32], int l)
    {
        constexpr int NS = kGridMaxBlocks / 32;
        const int nb = gridDim.x;
        unsigned long long *base = words + (size_t)2 * kGridCopies * nb * kGridWords;
        unsigned *count = reinterpret_cast<unsigned *>(base);
        T *slots = reinterpret_cast<T *>(base + 16) + (size_t)(fenced & 1u) * 2 * nb;
        ++fenced;
        if (l == 0) {
#pragma unroll
            for (int q = 0; q < NV; ++q) slots[q * nb + blockIdx.x] = s[q];
            fence();
            asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
            const unsigned want = fenced * (unsigned)nb;
            const long long t0 = clock64();
            for (;;) {
                unsigned v;
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
                if ((int)(v - want) >= 0) break;
                if (clock64() - t0 > limit) {
                    give_up();
                    break;
                }
            }
            fence();
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NV; ++q)
#pragma unroll
            for (int k = 0; k < NS; ++k) a[q][k] = l + 32 * k < nb ? ldcg(slots + q * nb + l + 32 * k) : T(0);
    }

    // v[q] = sum over the grid of v[q], q < NV (NV = 0: a barrier alone), then e[] = f(v)
    // (NX scalars: quotients are formed by one warp, an FP64 division by every thread
    // would hold the FP64 pipe for a microsecond); false once a wait gave up.  FENCED:
    // writes before the call by any thread of the grid are visible after it.
    template <class T, int NV, int NX, bool FENCED, class F> __device__ __forceinline__ bool sums(T *v, T *e, F f)
    {
        static_assert(NV <= 2 && NV + NX <= 4 && (NV > 0 || FENCED), "slots");
        const int tid = threadIdx.x, w = tid >> 5, l = tid & 31, nt = blockDim.x;
        T *bt = reinterpret_cast<T *>(buf);
        T *tot = reinterpret_cast<T *>(total);
        if constexpr (!FENCED) ++epoch;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if constexpr (sizeof(T) == 8) {
                bt[q * kGridBlockMax + tid] = v[q];
            } else {
                const T s = warp_sum(v[q]);
                if (l == 0) bt[q * kGridBlockMax + w] = s;
            }
        }
        __syncthreads();
        if (w == 0) {
            constexpr int NQ = NV > 0 ? NV : 1;
            T s[NQ], a[NQ][kGridMaxBlocks / 32];
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                const T *p = bt + q * kGridBlockMax;
                if constexpr (sizeof(T) == 8) {  // 64 clocks per dependent addition: four chains
                    T c[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) c[j] = l + 32 * j < nt ? p[l + 32 * j] : T(0);
                    for (int k = l + 128; k < nt; k += 128) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (k + 32 * j < nt) c[j] += p[k + 32 * j];
                    }
                    s[q] = (c[0] + c[1]) + (c[2] + c[3]);
                } else {
                    s[q] = l < (nt >> 5) ? p[l] : T(0);
                }
            }
#pragma unroll
            for (int q = 0; q < NV; ++q) s[q] = warp_sum(s[q]);
            if constexpr (FENCED) all_fenced<T, NV>(s, a, l);
            else all_tagged<T, NV>(s, a, l);
            if constexpr (NV > 0) {
                static_assert(kGridMaxBlocks / 32 == 5, "the tree below");
#pragma unroll
                for (int q = 0; q < NV; ++q) s[q] = ((a[q][0] + a[q][1]) + (a[q][2] + a[q][3])) + a[q][4];
#pragma unroll
                for (int q = 0; q < NV; ++q) s[q] = warp_sum(s[q]);
                T x[NX > 0 ? NX : 1];
                f(s, x);
                if (l == 0) {
#pragma unroll
                    for (int q = 0; q < NV; ++q) tot[q] = s[q];
#pragma unroll
                    for (int q = 0; q < NX; ++q) tot[NV + q] = x[q];
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = tot[q];
#pragma unroll
        for (int q = 0; q < NX; ++q) e[q] = tot[NV + q];
        return *s_dead == 0;
    }
    // sum and e = f(sum); the _pub forms also publish memory
    template <class T> __device__ __forceinline__ bool sum_pub(T &v)
    {
        return sums<T, 1, 0, true>(&v, static_cast<T *>(nullptr), [](const T *, T *) {});
    }
    template <class T> __device__ __forceinline__ bool sum(T &v)
    {
        return sums<T, 1, 0, false>(&v, static_cast<T *>(nullptr), [](const T *, T *) {});
    }
    template <class T, class F> __device__ __forceinline__ bool sum(T &v, T &e, F f)
    {
        return sums<T, 1, 1, false>(&v, &e, [&](const T *s, T *x) { x[0] = f(s[0]); });
    }
    template <class T, class F> __device__ __forceinline__ bool sum2(T &v, T &u, T &e, F f)
    {
        T a[2] = {v, u};
        const bool ok = sums<T, 2, 1, false>(a, &e, [&](const T *s, T *x) { x[0] = f(s[0], s[1]); });
        v = a[0];
        u = a[1];
        return ok;
    }
    __device__ __forceinline__ bool sync()
    {
        float *none = nullptr;
        return sums<float, 0, 0, true>(none, none, [](const float *, float *) {});
    }
};

// 64-bit words of the communication area: tagged slots [2][copies][blocks][kGridWords] | arrival
// count (128 bytes) | plain slots [2][2][blocks]
constexpr size_t grid_words(int blocks)
{
    return (size_t)2 * kGridCopies * blocks * kGridWords + 16 + (size_t)4 * blocks;
}

// sum of val[k] x[col[k]] over one row's entries: index order, one FMA per
// entry, up to eight gathers in flight
template <class T, class V>
__device__ __forceinline__ T slice_dot(const int *col, const V *val, int len, const T *x)
{
    T s = T(0);
    int k = 0;
    for (; k + 8 <= len; k += 8) {
        T v[8], g[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) g[u] = x[col[k + u]];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = (T)val[k + u];
#pragma unroll
        for (int u = 0; u < 8; ++u) s = fma(v[u], g[u], s);
    }
    const int rem = len - k;
    if (rem > 0) {  // 1 .. 7: gathers issued together, FMAs only for the row's entries
        T v[7], g[7];
#pragma unroll
        for (int u = 0; u < 7; ++u) {
            g[u] = u < rem ? x[col[k + u]] : T(0);
            v[u] = u < rem ? (T)val[k + u] : T(0);
        }
        if (rem & 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) s = fma(v[u], g[u], s);
            v[0] = v[4]; v[1] = v[5]; v[2] = v[6];
            g[0] = g[4]; g[1] = g[5]; g[2] = g[6];
        }
        if (rem & 2) {
            s = fma(v[0], g[0], s);
            s = fma(v[1], g[1], s);
            v[0] = v[2];
            g[0] = g[2];
        }
        if (rem & 1) s = fma(v[0], g[0], s);
    }
    return s;
}

// the same in FP64 with values `stride` apart (ELL keeps a row's values a slab apart)
__device__ __forceinline__ double slice_dot64(const int *col, const double *val, int64_t stride, int len, const double *x)
{
    if (stride == 1) return slice_dot<double, double>(col, val, len, x);
    double s = 0.0;
    for (int k = 0; k < len; ++k) s = fma(val[k * stride], x[col[k]], s);
    return s;
}

// first entry of row i (i <= n) in row-sorted COO
__device__ __forceinline__ int coo_row_start(const int *__restrict__ crow, int nnz, int i)
{
    int lo = 0, hi = nnz;
    while (lo < hi) {
        const int mid = lo + ((hi - lo) >> 1);
        if (crow[mid] < i) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// This thread's rows: u-th row lo + tid + u blockDim, its entries at [at, at + len) of the slice.
template <int R> struct GridRows {
    int at[R], len[R], row[R];  // row: -1 past the block's rows
};

// The solvers' results; kDead: a wait gave up.
constexpr int kDead = -1;

#define SPX_EACH(u) _Pragma("unroll") for (int u = 0; u < R; ++u) if (G.row[u] >= 0)
#define SPX_LIVE(call) \
    do {               \
        if (!(call)) return kDead; \
    } while (0)

// CG, the recurrence of cg_iter.  x: the iterate (registers); r: on entry the
// residual.  Ends with a status; iters and last (||r||^2) go on from the caller's.
// PRE (here and below): Jacobi, di the rows' M^-1.
template <class T, class V, int R, bool PRE>
__device__ __forceinline__ int grid_cg(GridTeam &tm, const GridRows<R> &G, const int *sc, const V *sv, T *ps, T (&x)[R],
                                       T (&r)[R], const T (&di)[R], T rho, T tol2, long long maxit, long long &iters,
                                       T &last)
{
    T p[R], q[R];
    last = rho;
    if (rho <= tol2) return SPX_CONVERGED;
    if (iters >= maxit) return SPX_MAX_ITER;
    if constexpr (PRE) rho = T(0);
    SPX_EACH(u)
    {
        p[u] = PRE ? di[u] * r[u] : r[u];
        ps[G.row[u]] = p[u];
        if constexpr (PRE) rho = fma(r[u], p[u], rho);
    }
    if constexpr (PRE) {  // r.z; also publishes p
        SPX_LIVE(tm.sum_pub(rho));
        if (rho == T(0)) return SPX_BREAKDOWN;
    } else {
        SPX_LIVE(tm.sync());
    }
    for (;;) {
        T pq = T(0);
        SPX_EACH(u)
        {
            q[u] = slice_dot<T, V>(sc + G.at[u], sv + G.at[u], G.len[u], ps);
            pq = fma(p[u], q[u], pq);
        }
        T alpha;
        SPX_LIVE(tm.sum(pq, alpha, [=](T s) { return rho / s; }));
        if (pq == T(0)) return SPX_BREAKDOWN;
        T rr = T(0), rz = T(0);
        SPX_EACH(u)
        {
            r[u] = fma(-alpha, q[u], r[u]);
            rr = fma(r[u], r[u], rr);
            if constexpr (PRE) rz = fma(r[u], di[u] * r[u], rz);
            x[u] = fma(alpha, p[u], x[u]);
        }
        T beta;
        if constexpr (PRE) SPX_LIVE(tm.sum2(rr, rz, beta, [=](T, T c) { return c / rho; }));
        else SPX_LIVE(tm.sum(rr, beta, [=](T s) { return s / rho; }));
        ++iters;
        last = rr;
        if (rr <= tol2) return SPX_CONVERGED;
        if (iters >= maxit) return SPX_MAX_ITER;
        if (PRE && rz == T(0)) return SPX_BREAKDOWN;
        rho = PRE ? rz : rr;
        SPX_EACH(u)
        {
            p[u] = fma(beta, p[u], PRE ? di[u] * r[u] : r[u]);
            ps[G.row[u]] = p[u];
        }
        SPX_LIVE(tm.sync());
    }
}

// BiCGSTAB, the recurrence of bi_iter (r^ = the residual on entry)
template <class T, class V, int R, bool PRE>
__device__ __forceinline__ int grid_bicgstab(GridTeam &tm, const GridRows<R> &G, const int *sc, const V *sv, T *ps,
                                             T (&x)[R], T (&r)[R], const T (&di)[R], T rho, T tol2, long long maxit,
                                             long long &iters, T &last)
{
    T rh[R], p[R], v[R];
    last = rho;
    if (rho <= tol2) return SPX_CONVERGED;
    if (iters >= maxit) return SPX_MAX_ITER;
    SPX_EACH(u)
    {
        rh[u] = r[u];
        p[u] = r[u];
        ps[G.row[u]] = PRE ? di[u] * r[u] : r[u];
    }
    SPX_LIVE(tm.sync());
    for (;;) {
        T rv = T(0);
        SPX_EACH(u)
        {
            v[u] = slice_dot<T, V>(sc + G.at[u], sv + G.at[u], G.len[u], ps);
            rv = fma(rh[u], v[u], rv);
        }
        T alpha;
        SPX_LIVE(tm.sum(rv, alpha, [=](T s) { return rho / s; }));
        if (rv == T(0)) return SPX_BREAKDOWN;
        T ss = T(0);
        SPX_EACH(u)
        {
            r[u] = fma(-alpha, v[u], r[u]);  // s, in r's place
            ps[G.row[u]] = PRE ? di[u] * r[u] : r[u];
            ss = fma(r[u], r[u], ss);
        }
        SPX_LIVE(tm.sum_pub(ss));
        ++iters;
        if (ss <= tol2) {
            SPX_EACH(u) x[u] = fma(alpha, PRE ? di[u] * p[u] : p[u], x[u]);
            last = ss;
            return SPX_CONVERGED;
        }
        T t[R], ts = T(0), tt = T(0);
        SPX_EACH(u)
        {
            t[u] = slice_dot<T, V>(sc + G.at[u], sv + G.at[u], G.len[u], ps);
            ts = fma(r[u], t[u], ts);
            tt = fma(t[u], t[u], tt);
        }
        T omega;
        SPX_LIVE(tm.sum2(ts, tt, omega, [](T a, T c) { return a / c; }));
        if (tt == T(0)) return SPX_BREAKDOWN;
        T rr = T(0), rhr = T(0);
        SPX_EACH(u)
        {
            x[u] = PRE ? fma(omega, di[u] * r[u], fma(alpha, di[u] * p[u], x[u]))
                       : fma(omega, r[u], fma(alpha, p[u], x[u]));
            r[u] = fma(-omega, t[u], r[u]);
            rr = fma(r[u], r[u], rr);
            rhr = fma(rh[u], r[u], rhr);
        }
        T beta;
        SPX_LIVE(tm.sum2(rr, rhr, beta, [=](T, T c) { return (c / rho) * (alpha / omega); }));
        last = rr;
        if (rr <= tol2) return SPX_CONVERGED;
        if (omega == T(0)) return SPX_BREAKDOWN;
        if (iters >= maxit) return SPX_MAX_ITER;
        if (rhr == T(0)) return SPX_BREAKDOWN;
        rho = rhr;
        SPX_EACH(u)
        {
            p[u] = fma(beta, fma(-omega, v[u], p[u]), r[u]);
            ps[G.row[u]] = PRE ? di[u] * p[u] : p[u];
        }
        SPX_LIVE(tm.sync());
    }
}

// CGS, the recurrence of cgs_iter (r^ = the residual on entry).  stall > 0: the
// inner cycle's stall rule.
template <class T, class V, int R, bool PRE>
__device__ __forceinline__ int grid_cgs(GridTeam &tm, const GridRows<R> &G, const int *sc, const V *sv, T *ps, T (&x)[R],
                                        T (&r)[R], const T (&di)[R], T rho, T bb, T tol2, long long maxit, int stall,
                                        long long &iters, T &last)
{
    T rh[R], p[R], uu[R], q[R];
    T mark = T(1);
    long long mark_it = 0, it = 0;
    last = rho;
    if (rho <= tol2) return SPX_CONVERGED;
    if (iters >= maxit) return SPX_MAX_ITER;
    SPX_EACH(u)
    {
        rh[u] = p[u] = uu[u] = r[u];
        ps[G.row[u]] = PRE ? di[u] * r[u] : r[u];
    }
    SPX_LIVE(tm.sync());
    for (;;) {
        T rv = T(0);
        SPX_EACH(u)
        {
            q[u] = slice_dot<T, V>(sc + G.at[u], sv + G.at[u], G.len[u], ps);  // v = A p
            rv = fma(rh[u], q[u], rv);
        }
        T alpha;
        SPX_LIVE(tm.sum(rv, alpha, [=](T s) { return rho / s; }));
        if (rv == T(0)) return SPX_BREAKDOWN;
        SPX_EACH(u)
        {
            q[u] = fma(-alpha, q[u], uu[u]);
            const T w = PRE ? di[u] * (uu[u] + q[u]) : uu[u] + q[u];
            x[u] = fma(alpha, w, x[u]);
            ps[G.row[u]] = w;
        }
        SPX_LIVE(tm.sync());
        T rr = T(0), rhr = T(0);
        SPX_EACH(u)
        {
            r[u] = fma(-alpha, slice_dot<T, V>(sc + G.at[u], sv + G.at[u], G.len[u], ps), r[u]);
            rr = fma(r[u], r[u], rr);
            rhr = fma(rh[u], r[u], rhr);
        }
        T beta;
        SPX_LIVE(tm.sum2(rr, rhr, beta, [=](T, T c) { return c / rho; }));
        ++iters;
        ++it;
        last = rr;
        if (rr <= tol2) return SPX_CONVERGED;
        if (iters >= maxit) return SPX_MAX_ITER;
        if (stall > 0) {
            const T rel = sqrt(rr / bb);
            if (rel < T(0.5) * mark) {
                mark = rel;
                mark_it = it;
            } else if (it - mark_it >= stall) {
                return SPX_STAGNATED;
            }
        }
        if (rhr == T(0)) return SPX_BREAKDOWN;
        rho = rhr;
        SPX_EACH(u)
        {
            uu[u] = fma(beta, q[u], r[u]);
            p[u] = fma(beta, fma(beta, p[u], q[u]), uu[u]);
            ps[G.row[u]] = PRE ? di[u] * p[u] : p[u];
        }
        SPX_LIVE(tm.sync());
    }
}

// One solve in one precision: b = 0, restarts from the true residual (run_short's policy)
template <class T, int SOLVER, int R, bool PRE>
__device__ __forceinline__ int grid_solve_one(GridTeam &tm, const GridRows<R> &G, const int *sc, const T *sv,
                                              const T (&di)[R], const GridArgs &A, GridOut &o)
{
    const T *b = static_cast<const T *>(A.b);
    T *xg = static_cast<T *>(A.x), *ps = static_cast<T *>(A.ps);
    T x[R], r[R], bb = T(0);
    SPX_EACH(u)
    {
        const T bi = b[G.row[u]];
        bb = fma(bi, bi, bb);
        x[u] = xg[G.row[u]];
        ps[G.row[u]] = x[u];
    }
    SPX_LIVE(tm.sum_pub(bb));
    if (bb == T(0)) {
        SPX_EACH(u) xg[G.row[u]] = T(0);
        o.status = SPX_CONVERGED;
        return 0;
    }
    const T tol2 = (T)(A.tol * A.tol) * bb;
    // r = b - A x (x published in ps), ||r||^2
    auto residual = [&](T &rr) -> bool {
        rr = T(0);
        SPX_EACH(u)
        {
            r[u] = b[G.row[u]] - slice_dot<T, T>(sc + G.at[u], sv + G.at[u], G.len[u], ps);
            rr = fma(r[u], r[u], rr);
        }
        return tm.sum(rr);
    };
    T rr;
    SPX_LIVE(residual(rr));
    for (;;) {
        T last;
        int st;
        if constexpr (SOLVER == SPX_CG)
            st = grid_cg<T, T, R, PRE>(tm, G, sc, sv, ps, x, r, di, rr, tol2, A.maxit, o.iters, last);
        else if constexpr (SOLVER == SPX_CGS)
            st = grid_cgs<T, T, R, PRE>(tm, G, sc, sv, ps, x, r, di, rr, bb, tol2, A.maxit, 0, o.iters, last);
        else st = grid_bicgstab<T, T, R, PRE>(tm, G, sc, sv, ps, x, r, di, rr, tol2, A.maxit, o.iters, last);
        if (st == kDead) return kDead;
        o.status = st;
        o.relres = (double)sqrt(last / bb);
        // the true residual; every gather of ps ended before the last sum of the solver
        SPX_EACH(u) ps[G.row[u]] = x[u];
        SPX_LIVE(tm.sync());
        SPX_LIVE(residual(rr));
        o.relres_true = sqrt((double)rr / (double)bb);
        if (st != SPX_CONVERGED || o.relres_true <= A.tol) break;
        if (o.restarts == kGridRestarts) {
            o.status = SPX_STAGNATED;
            break;
        }
        ++o.restarts;
    }
    SPX_EACH(u) xg[G.row[u]] = x[u];
    return 0;
}

// Mixed precision: CG with reliable updates (run_cg_reliable's policy), BiCGSTAB,
// CGS and preconditioned CG as FP64 refinement (run_ir's policy).  sv: FP32 values; the FP64
// residual reads the FP64 values from global memory.
template <int SOLVER, int R, bool PRE>
__device__ __forceinline__ int grid_solve_mixed(GridTeam &tm, const GridRows<R> &G, const int *sc, const float *sv,
                                                const float (&di)[R], const GridArgs &A, int j0, GridOut &o)
{
    const double *b = static_cast<const double *>(A.b);
    const double *v64 = static_cast<const double *>(A.val64) + j0;  // (ELL: j0 = 0, a row's values ell_ld apart)
    double *xg = static_cast<double *>(A.x);
    float *ps = static_cast<float *>(A.ps);
    double x[R], r64[R], bb = 0.0;
    SPX_EACH(u)
    {
        const double bi = b[G.row[u]];
        bb = fma(bi, bi, bb);
        x[u] = xg[G.row[u]];
    }
    SPX_LIVE(tm.sum(bb));
    if (bb == 0.0) {
        SPX_EACH(u) xg[G.row[u]] = 0.0;
        o.status = SPX_CONVERGED;
        return 0;
    }
    double rr64;
    // r64 = b - A x in FP64, ||r64||^2
    auto residual64 = [&]() -> bool {
        SPX_EACH(u) A.xs[G.row[u]] = x[u];
        if (!tm.sync()) return false;
        rr64 = 0.0;
        SPX_EACH(u)
        {
            const double *v = A.ell_ld ? v64 + G.row[u] : v64 + G.at[u];
            r64[u] = b[G.row[u]] - slice_dot64(sc + G.at[u], v, A.ell_ld ? A.ell_ld : 1, G.len[u], A.xs);
            rr64 = fma(r64[u], r64[u], rr64);
        }
        return tm.sum(rr64);
    };
    SPX_LIVE(residual64());
    if constexpr (SOLVER == SPX_CG && !PRE) {
        o.relres = sqrt(rr64 / bb);
        o.status = o.relres <= A.tol ? SPX_CONVERGED : SPX_MAX_ITER;
        if (o.status != SPX_CONVERGED) {
            const float tol2 = (float)(A.tol * A.tol * bb);
            float d[R], r[R], p[R], q[R], rho = 0.f;
            SPX_EACH(u)
            {
                r[u] = (float)r64[u];
                p[u] = r[u];
                d[u] = 0.f;
                ps[G.row[u]] = p[u];
                rho = fmaf(r[u], r[u], rho);
            }
            SPX_LIVE(tm.sum_pub(rho));  // also publishes p
            float maxr2 = rho;
            int st = o.iters >= A.maxit ? SPX_MAX_ITER : SPX_CONVERGED;
            bool go = st == SPX_CONVERGED;
            for (;;) {
                float rr = 0.f;
                while (go) {
                    float pq = 0.f;
                    SPX_EACH(u)
                    {
                        q[u] = slice_dot<float, float>(sc + G.at[u], sv + G.at[u], G.len[u], ps);
                        pq = fmaf(p[u], q[u], pq);
                    }
                    float alpha;
                    SPX_LIVE(tm.sum(pq, alpha, [=](float s) { return rho / s; }));
                    if (pq == 0.f) {
                        st = SPX_BREAKDOWN;
                        break;
                    }
                    rr = 0.f;
                    SPX_EACH(u)
                    {
                        r[u] = fmaf(-alpha, q[u], r[u]);
                        rr = fmaf(r[u], r[u], rr);
                        d[u] = fmaf(alpha, p[u], d[u]);
                    }
                    float beta;
                    SPX_LIVE(tm.sum(rr, beta, [=](float s) { return s / rho; }));
                    ++o.iters;
                    if (rr <= tol2) break;
                    if (o.iters >= A.maxit) {
                        st = SPX_MAX_ITER;
                        break;
                    }
                    if (rr > maxr2) maxr2 = rr;
                    if (rr < kGridRuDelta2 * maxr2) break;
                    rho = rr;
                    SPX_EACH(u)
                    {
                        p[u] = fmaf(beta, p[u], r[u]);
                        ps[G.row[u]] = p[u];
                    }
                    SPX_LIVE(tm.sync());
                }
                // reliable update: x += d, the residual again in FP64
                SPX_EACH(u)
                {
                    x[u] += (double)d[u];
                    d[u] = 0.f;
                }
                SPX_LIVE(residual64());
                ++o.restarts;
                o.relres = sqrt(rr64 / bb);
                if (o.relres <= A.tol) {
                    o.status = SPX_CONVERGED;
                    break;
                }
                if (st != SPX_CONVERGED) {  // the budget is spent, or the iteration broke down
                    o.status = st;
                    break;
                }
                // the rounding of the FP64 residual replaces r; beta with it; p = r + beta p
                float r2 = 0.f;
                SPX_EACH(u)
                {
                    r[u] = (float)r64[u];
                    r2 = fmaf(r[u], r[u], r2);
                }
                SPX_LIVE(tm.sum(r2));
                const float beta = r2 / rho;
                rho = maxr2 = r2;
                if (o.iters >= A.maxit) {  // the iteration that met tol in FP32 was the last allowed
                    st = SPX_MAX_ITER;
                    go = false;
                }
                SPX_EACH(u)
                {
                    p[u] = fmaf(beta, p[u], r[u]);
                    ps[G.row[u]] = p[u];
                }
                SPX_LIVE(tm.sync());
            }
        }
    } else {
        o.status = SPX_MAX_ITER;
        for (;; ++o.restarts) {
            const double rn = sqrt(rr64);
            o.relres = rn / sqrt(bb);
            if (o.relres <= A.tol) {
                o.status = SPX_CONVERGED;
                break;
            }
            if (o.restarts >= 20 || o.iters >= A.maxit) break;
            // A32 d = r / ||r|| to 1e-4, d from 0
            const double scale = 1.0 / rn;
            float r[R], d[R], bb32 = 0.f, last;
            SPX_EACH(u)
            {
                r[u] = (float)(r64[u] * scale);
                d[u] = 0.f;
                bb32 = fmaf(r[u], r[u], bb32);
            }
            SPX_LIVE(tm.sum(bb32));
            int st = SPX_CONVERGED;
            if (bb32 != 0.f) {
                const float tol2 = (float)(1e-4 * 1e-4) * bb32;
                const long long cyc = min(A.maxit - o.iters, (long long)kIrInnerCap);
                long long it = 0;
                if constexpr (SOLVER == SPX_CGS)
                    st = grid_cgs<float, float, R, PRE>(tm, G, sc, sv, ps, d, r, di, bb32, bb32, tol2, cyc, kIrCgsStall,
                                                        it, last);
                else if constexpr (SOLVER == SPX_CG)
                    st = grid_cg<float, float, R, PRE>(tm, G, sc, sv, ps, d, r, di, bb32, tol2, cyc, it, last);
                else
                    st = grid_bicgstab<float, float, R, PRE>(tm, G, sc, sv, ps, d, r, di, bb32, tol2, cyc, it, last);
                o.iters += it;
            }
            if (st == kDead) return kDead;
            SPX_EACH(u) x[u] = fma(rn, (double)d[u], x[u]);
            SPX_LIVE(residual64());
        }
    }
    o.relres_true = o.relres;
    SPX_EACH(u) xg[G.row[u]] = x[u];
    return 0;
}

#undef SPX_EACH
#undef SPX_LIVE

// Shared memory: column indices | values | the sums' buffer
template <class V> constexpr size_t grid_smem(int cap)
{
    return ((size_t)cap * 4 + 15) / 16 * 16 + ((size_t)cap * sizeof(V) + 15) / 16 * 16 + 2 * kGridBlockMax * 8;
}

__device__ __forceinline__ void grid_error(const GridArgs &A, unsigned bits)
{
    atomicOr(A.err, bits);
    atomicOr(&A.out->err, bits);
}

// block 0: the result, err left to atomics
__device__ __forceinline__ void grid_report(const GridArgs &A, const GridOut &o)
{
    if (const unsigned before = ldcg(A.err)) grid_error(A, before);
    A.out->status = o.status;
    A.out->restarts = o.restarts;
    A.out->iters = o.iters;
    A.out->relres = o.relres;
    A.out->relres_true = o.relres_true;
    A.out->done = 1;
}

// T: the precision of b and x; V: of the values the products use (V = float, T = double: mixed).
// COMPACT: the same with at most 64 registers per thread, so that the solves of two contexts fit
// on an SM beside each other; the same operations in the same order, so the same bits.
template <class T, class V, int SOLVER, int R, bool PRE, bool COMPACT>
__global__ void __launch_bounds__(kGridBlockMax, COMPACT ? 2 : 1) k_grid_solve(GridArgs A)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ double total[4];
    __shared__ int s_dead;
    int *sc = reinterpret_cast<int *>(smem);
    V *sv = reinterpret_cast<V *>(smem + ((size_t)A.cap * 4 + 15) / 16 * 16);
    GridTeam tm;
    tm.words = A.words;
    tm.buf = reinterpret_cast<double *>(reinterpret_cast<unsigned char *>(sv) + ((size_t)A.cap * sizeof(V) + 15) / 16 * 16);
    tm.total = total;
    tm.s_dead = &s_dead;
    const int tid = threadIdx.x, nt = blockDim.x;
    if (tid == 0) s_dead = 0;
    const int lo = min(A.n, (int)blockIdx.x * A.rows), hi = min(A.n, lo + A.rows);
    const V *val = static_cast<const V *>(A.val);
    GridRows<R> G;
    int j0 = 0;
    bool fits = true;
    if (A.ell_ld) {
        // a row's entries fill its first slots; row lo + q goes to the slice at q ell_w
        fits = (hi - lo) * A.ell_w <= A.cap;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int q = tid + u * nt, i = lo + q;
            G.row[u] = i < hi ? i : -1;
            G.at[u] = q * A.ell_w;
            G.len[u] = 0;
            if (i >= hi || !fits) continue;
            for (int k = 0; k < A.ell_w; ++k) {
                const int c = A.col[k * A.ell_ld + i];
                if (c < 0) break;
                sc[G.at[u] + k] = c;
                sv[G.at[u] + k] = val[k * A.ell_ld + i];
                G.len[u] = k + 1;
            }
        }
    } else {
        auto start = [&](int i) { return A.crow ? coo_row_start(A.crow, A.nnz, i) : A.rp[i]; };
        j0 = start(lo);
        const int nz = start(hi) - j0;
        fits = nz <= A.cap;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const int i = lo + tid + u * nt;
            G.row[u] = i < hi ? i : -1;
            G.at[u] = i < hi ? start(i) - j0 : 0;
            G.len[u] = i < hi && fits ? start(i + 1) - j0 - G.at[u] : 0;
        }
        if (fits)
            for (int k = tid; k < nz; k += nt) {
                sc[k] = A.col[j0 + k];
                sv[k] = val[j0 + k];
            }
    }
    if (!fits && tid == 0) grid_error(A, DEVERR_BOUNDS);  // never, for the matrix the slice was sized for
    __syncthreads();
    // M^-1 = 1 / (the sum of the row's diagonal entries), 1 where that is 0 (k_jacobi_dinv's rule, from
    // the matrix's own values)
    V di[R];
    if constexpr (PRE) {
#pragma unroll
        for (int u = 0; u < R; ++u) {
            double d = 0.0;
            for (int k = 0; k < G.len[u]; ++k)
                if (sc[G.at[u] + k] == G.row[u]) {
                    if constexpr (sizeof(T) == sizeof(V)) {
                        d += (double)sv[G.at[u] + k];
                    } else {
                        const double *v64 = static_cast<const double *>(A.val64);
                        d += A.ell_ld ? v64[k * A.ell_ld + G.row[u]] : v64[j0 + G.at[u] + k];
                    }
                }
            di[u] = d != 0.0 ? (V)(1.0 / d) : V(1);
        }
    }
    GridOut o{1, SPX_MAX_ITER, 0, 0u, 0, 0.0, 0.0};
    int st;
    if constexpr (sizeof(T) != sizeof(V)) st = grid_solve_mixed<SOLVER, R, PRE>(tm, G, sc, sv, di, A, j0, o);
    else st = grid_solve_one<T, SOLVER, R, PRE>(tm, G, sc, sv, di, A, o);
    if (st == kDead && tid == 0) grid_error(A, DEVERR_QUEUE_TIMEOUT);
    if (st != kDead && blockIdx.x == 0 && tid == 0) grid_report(A, o);
}

// Launch of one (T, V, COMPACT): grid_f64.cu, grid_f32.cu, grid_mixed.cu and their _compact
// forms.  SPX_ERR_UNSUPPORTED when the device cannot hold the grid at once.
template <class T, class V, int SOLVER, int R, bool PRE, bool COMPACT>
int grid_launch_r(spx_ctx *ctx, const GridArgs &A, int blocks, int threads)
{
    auto kern = k_grid_solve<T, V, SOLVER, R, PRE, COMPACT>;
    const size_t smem = grid_smem<V>(A.cap);
    int lim = 0;
    SPX_TRY(smem_optin(reinterpret_cast<const void *>(kern), -1, &lim));
    if (smem > (size_t)lim) return SPX_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, A);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        return SPX_ERR_UNSUPPORTED;
    }
    return e == cudaSuccess ? SPX_OK : cuda_fail(e, "cudaLaunchKernelEx(k_grid_solve)");
}

template <class T, class V, int SOLVER, bool PRE, bool COMPACT>
int grid_launch_s(spx_ctx *ctx, const GridArgs &A, int blocks, int threads, int r)
{
    if (r == 1) return grid_launch_r<T, V, SOLVER, 1, PRE, COMPACT>(ctx, A, blocks, threads);
    if (r == 2) return grid_launch_r<T, V, SOLVER, 2, PRE, COMPACT>(ctx, A, blocks, threads);
    if constexpr (COMPACT && sizeof(V) == 8) return SPX_ERR_UNSUPPORTED;  // (spills: no gain)
    else return grid_launch_r<T, V, SOLVER, 4, PRE, COMPACT>(ctx, A, blocks, threads);
}

template <class T, class V, bool PRE, bool COMPACT>
int grid_launch(spx_ctx *ctx, const GridArgs &A, int solver, int blocks, int threads, int r)
{
    if (solver == SPX_CG) return grid_launch_s<T, V, SPX_CG, PRE, COMPACT>(ctx, A, blocks, threads, r);
    if (solver == SPX_CGS) return grid_launch_s<T, V, SPX_CGS, PRE, COMPACT>(ctx, A, blocks, threads, r);
    return grid_launch_s<T, V, SPX_BICGSTAB, PRE, COMPACT>(ctx, A, blocks, threads, r);
}

}  // namespace spx
