// Shared device helpers of the Radsort CUDA library (sm_103a).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "rs_kernels.cuh"

namespace rs {

// ---------------------------------------------------------------- status
// Sticky device status word (bit set = error class seen); read and cleared by
// radsort_device_status().  Kernels never trap: they record and return.
// One word per translation unit (no relocatable device code needed); each
// unit exports a host function that reads and clears its word.
static __device__ unsigned g_status = 0;

static inline unsigned take_status_word()
{
    unsigned v = 0, zero = 0;
    if (cudaMemcpyFromSymbol(&v, g_status, sizeof(v)) != cudaSuccess)
        return ST_INTERNAL;
    cudaMemcpyToSymbol(g_status, &zero, sizeof(zero));
    return v;
}

__device__ __forceinline__ void set_status(unsigned bits) { atomicOr(&g_status, bits); }

// Iteration limit of every spin-wait (each iteration sleeps >= 64 ns, so the
// limit is several seconds of wall time on a healthy GPU).
constexpr unsigned SPIN_LIMIT = 1u << 26;

// True once any wait of this translation unit has run out: the other waits
// give up at their next check instead of running out one after another.
__device__ __forceinline__ bool wait_failed()
{
    return (*reinterpret_cast<volatile unsigned *>(&g_status) & ST_TIMEOUT) != 0;
}

// ---------------------------------------------------------------- smem / mbarrier / bulk copy
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase with the given parity to complete.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity)
{
    for (unsigned it = 0; it < SPIN_LIMIT; ++it) {
        if (mbar_try_wait(bar, parity))
            return true;
        if ((it & 1023u) == 1023u && wait_failed())
            return false;
        __nanosleep(64);
    }
    set_status(ST_TIMEOUT);
    return false;
}

// Orders this thread's earlier generic-proxy accesses to shared memory before
// later async-proxy (bulk copy) accesses to the same bytes.  Every thread that
// read or wrote a buffer with plain loads and stores executes it before the
// barrier / mbarrier arrive that hands the buffer back to a bulk-copy issuer.
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// The same for memory in general: before bulk copies that read global memory
// written with plain stores.
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

// 1-D bulk copy global -> shared through the TMA engine; completion is
// signalled on `bar` as transaction bytes.  dst, src and bytes must be
// multiples of 16.
__device__ __forceinline__ void bulk_g2s(void *dst_smem, const void *src_gmem, uint32_t bytes,
                                         uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst_smem)),
        "l"(src_gmem), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// ---------------------------------------------------------------- warp / block scans
__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

template <typename T> __device__ __forceinline__ T warp_incl_scan(T v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o)
            v += t;
    }
    return v;
}

template <typename T> __device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Named barrier over the first `nthreads` threads of the block (id != 0).
__device__ __forceinline__ void named_bar(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Arrival without waiting at named barrier `id` (its other threads wait).
__device__ __forceinline__ void bar_arrive(int id, int nthreads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Mask of the lanes whose digit equals this lane's, among lanes with
// `valid` set: one ballot per digit bit (warp-level multisplit).  All 32
// lanes must call it.
template <int DB> __device__ __forceinline__ unsigned peer_mask(uint32_t d, bool valid)
{
    unsigned m = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int bit = 0; bit < DB; ++bit) {
        const bool on = (d >> bit) & 1u;
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        m &= on ? bal : ~bal;
    }
    return m;
}

// Stable ranks of a half-warp's elements, ITEMS rows of 16: row holds a zeroed
// word per digit, the count so far in its high half and the lanes of the
// present row in its low half.  Lanes with the same digit OR their bit into the
// digit's word and read it back; the last of them writes the new count (its
// rank + 1) with the lane bits cleared.  digit(it): this lane's digit in row
// it; real(it): whether it has an element there (missing ones come last).
// rk: two 16-bit ranks a word.  All 32 lanes call it, each half with its row.
template <int ITEMS, typename D, typename V>
__device__ __forceinline__ void rank_half_warp(uint32_t *row, D &&digit, V &&real, uint32_t (&rk)[(ITEMS + 1) / 2])
{
    const uint32_t l16 = threadIdx.x & 15u, ltm = (1u << l16) - 1u, gtm = 0xFFFFu & ~((2u << l16) - 1u);
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        uint32_t *w = row + digit(it);
        if (real(it))
            atomicOr(w, 1u << l16);
        __syncwarp();
        const uint32_t v = *reinterpret_cast<volatile uint32_t *>(w);
        const uint32_t r = (v >> 16) + __popc(v & ltm);
        __syncwarp();
        if (real(it) && !(v & gtm))
            *reinterpret_cast<volatile uint32_t *>(w) = (r + 1u) << 16;
        __syncwarp();
        if (it & 1)
            rk[it >> 1] |= r << 16;
        else
            rk[it >> 1] = r;
    }
}

// ---------------------------------------------------------------- thread-block clusters
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// every thread of the cluster; orders shared-memory accesses across its CTAs
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// this shared-memory address in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// 64 bits that another CTA may be storing meanwhile (st_relaxed64): relaxed
// accesses that cover each other whole are single-copy atomic, so the load
// returns one of the values stored; of a weak load that races with a store the
// memory model says nothing, it may be half of each
__device__ __forceinline__ unsigned long long ld_relaxed64(uint32_t addr)
{
    unsigned long long v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed64(uint32_t addr, unsigned long long v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t add_cluster(uint32_t addr, uint32_t v)
{
    uint32_t r;
    asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(r) : "r"(addr), "r"(v) : "memory");
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t addr, uint2 v)
{
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}

// ---------------------------------------------------------------- keys
template <typename KT> __device__ __forceinline__ uint32_t digit_of(KT k, uint32_t shift,
                                                                     uint32_t mask)
{
    return static_cast<uint32_t>(k >> shift) & mask;
}

// IEEE float32 bits <-> unsigned-orderable bits: the sign bit of non-negative
// values flips, every bit of negative ones
__device__ __forceinline__ uint32_t float_to_ordered(uint32_t x) { return x ^ ((x >> 31) ? 0xFFFFFFFFu : 0x80000000u); }
__device__ __forceinline__ uint32_t ordered_to_float(uint32_t x) { return x ^ ((x >> 31) ? 0x80000000u : 0xFFFFFFFFu); }

} // namespace rs
