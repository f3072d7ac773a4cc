// dev_common.cuh -- device helpers: deterministic reductions, last-block
// detection, mbarrier + 1-D bulk (TMA) copies with bounded waits.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "spx_internal.cuh"

namespace spx {

// ------------------------------------------------------------------ reductions
// Fixed shuffle pattern => the same inputs always give the same bits.
template <class T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int warp_max(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Lane l of one warp adds buf[l], buf[l + 32], ... (index order, four partial
// sums) and the warp adds the lanes' sums; valid in every lane.
template <class T, int NW> __device__ __forceinline__ T strided_sum(const T *buf, int l)
{
    constexpr int Q = NW < 4 ? NW : 4;
    T a[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) a[q] = buf[l + 32 * q];
#pragma unroll
    for (int k = Q; k < NW; ++k) a[k % Q] += buf[l + 32 * k];
#pragma unroll
    for (int q = 1; q < Q; ++q) a[0] += a[q];
    return warp_sum(a[0]);
}

// Sums of NV values over the block, valid in every thread.  Two barriers; the
// callers' earlier shared-memory accesses are ordered before the first.
//
// FP64: the values go through shared memory and one warp per sum adds them,
// BLOCK/32 - 1 additions and 5 shuffle steps.  GB300's two FP64 lanes per SM
// make every FP64 warp instruction cost 16 clocks, so a shuffle tree in every
// warp (5 BLOCK/32 + 5 additions, most lanes of them redundant) held the pipe
// for as long as a row of FMAs per thread.  With this and unused sums left
// out, an FP64 CG iteration on 128^3 took 70.2 us against 75.0 us, BiCGSTAB on
// 30 001 rows of 20 random columns 1.42 ms against 1.64 ms, block-Jacobi
// BiCGSTAB on 101^3 24.1 against 26.5 ms and a batch of 4096 systems 30.8
// against 31.7 ms.  FP32 shuffles are cheap and keep the tree.
// buf: NV BLOCK elements of shared memory for the FP64 sums (block_sums_in: the
// caller's, free for the block to overwrite; block_sums: its own).
template <class T, int BLOCK, int NV> __device__ __forceinline__ void block_sums_in(T (&v)[NV], T *buf)
{
    static_assert(BLOCK % 32 == 0 && BLOCK <= 1024, "block size");
    constexpr int NW = BLOCK / 32;
    __shared__ T total[NV];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int q = 0; q < NV; ++q) buf[q * BLOCK + threadIdx.x] = v[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (w == q % NW) {
                const T s = strided_sum<T, NW>(buf + q * BLOCK, l);
                if (l == 0) total[q] = s;
            }
    } else {
        __shared__ T part[NV][NW];
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const T s = warp_sum(v[q]);
            if (l == 0) part[q][w] = s;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (w == q % NW) {
                const T s = warp_sum(l < NW ? part[q][l] : T(0));
                if (l == 0) total[q] = s;
            }
    }
    // a thread rewrites buf / part only past this barrier and total only past the
    // first barrier of the next call, when every thread has read it
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = total[q];
}

template <class T, int BLOCK, int NV> __device__ __forceinline__ void block_sums(T (&v)[NV])
{
    if constexpr (sizeof(T) == 8) {
        __shared__ T buf[NV * BLOCK];
        block_sums_in<T, BLOCK, NV>(v, buf);
    } else {
        block_sums_in<T, BLOCK, NV>(v, nullptr);
    }
}

template <class T, int BLOCK> __device__ __forceinline__ T block_sum(T v)
{
    T a[1] = {v};
    block_sums<T, BLOCK, 1>(a);
    return a[0];
}

// Last-block detection (threadfence reduction pattern).  Every block calls
// it once, after its global writes; it returns true in exactly one block, the
// last to arrive, which then sees all other blocks' writes.  The last block
// resets the counter for the next launch in stream order.
__device__ __forceinline__ bool last_block(unsigned *ticket, unsigned nblocks)
{
    __shared__ unsigned s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned prev = atomicAdd(ticket, 1u);
        s_last = (prev == nblocks - 1) ? 1u : 0u;
        if (s_last) *ticket = 0u;
    }
    __syncthreads();
    const bool last = s_last != 0u;
    if (last) __threadfence();
    return last;
}

// L1-bypassing loads for data written by other blocks of the same launch.
template <class T> __device__ __forceinline__ T ldcg(const T *p) { return __ldcg(p); }

// ------------------------------------------------------------------ mbarrier + bulk copy
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Order this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (bulk copy) writes to the same memory.
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

// 1-D bulk copy global -> shared, completion counted on `bar`.  dst, src and
// bytes must be multiples of 16 (the callers round ranges outwards inside
// padded allocations).
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// The same for data read once per launch (a matrix streamed past the vectors): its L2
// lines are the first to go, so the vectors of a solver iteration stay in the 129 MB
// (CG on 128^3, 184 MB of matrix and 67 MB of vectors: 70.2 -> 64.2 us per iteration;
// the 27-point product 100^3, whose x is 8 MB, 73.7 -> 72.8 us).
__device__ __forceinline__ uint64_t policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ void bulk_g2s_once(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0u;
}

// Bounded wait for phase `parity` of `bar`: gives up after about `limit_cycles`
// SM clock cycles, sets DEVERR_MBAR_TIMEOUT in *err and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, unsigned *err,
                                          long long limit_cycles = 2000000000LL)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit_cycles) {
            if (err) atomicOr(err, DEVERR_MBAR_TIMEOUT);
            return false;
        }
    }
    return true;
}

}  // namespace spx
