// Radsort rounds with one block chain per bucket for the whole array, and the
// out-of-place comparison sort (Alg. 1), on one pipelined round kernel for
// sm_103a.
//
// Grid layout of the block chains.  The paper's parallel variant (Sec. 4.3)
// gives every chunk its own head start and its own open block per bucket, so
// the scratch array grows with the chunk count (2*sigma*p blocks).  Here all
// CTAs share one free list and one chain per bucket, like the sequential
// algorithm (Alg. 5 with a head start of sigma blocks, Sec. 2.1), and the
// chains are laid on the block grid of the round's output: logical data block
// j holds output positions [j*b, (j+1)*b) of the stably sorted sequence.  A
// block that contains the start of a bucket (strictly inside) is shared by
// two or more buckets; every other block belongs to one bucket.
//   * The bucket sizes of every digit come from one upfront histogram pass
//     (the paper's "generic" variant, Sec. 5), so bucket c's output range
//     [O_c, O_c + n_c) and the shared blocks are known before a round.
//   * Before the round, the shared blocks (fewer than sigma) and the first
//     L = GRID_AHEAD non-shared blocks of every bucket take the first
//     nP < (L+1)*sigma free-list entries.
//   * A tile learns where its elements of bucket c go, O_c + E_c(t), from a
//     decoupled look-back over the per-bucket counts of earlier tiles.
//     Every other block j of bucket c is taken eagerly, as newBucketBlock
//     does in Alg. 5 but L blocks ahead: by the tile that writes the first
//     position of block j - L, at a free-list index in  nP + (blocks taken
//     by earlier tiles) + [0, blocks this tile takes); the count for earlier
//     tiles follows from E(t) alone, the order within the tile is free.  A tile that continues
//     a block therefore finds it taken long before (a bounded wait covers
//     the rest), and tiles in flight together do not wait on each other.
//   * The free list is the current logical order: (L+2)*sigma head-start
//     blocks, then the input blocks in order.  Tiles are dispatched in input
//     order, a tile reads its blocks before it publishes its counts, and
//     after the tiles up to t at most  nP + (elements)/b + sigma <
//     (L+2)*sigma + (blocks read)  blocks have been taken (Lemma 1 with a
//     head start of (L+2)*sigma).
//   * The tile that takes a block records it in the next block map pi',
//     where later tiles find it.
// The next round's head start is the (L+2)*sigma entries after the last
// taken one, so the scratch array holds (L+2)*sigma + 1 blocks whatever the
// number of CTAs, and after the last round every block but the array's tail
// is full: Finalize is a block permutation plus one tail copy.
//
// Round kernel (k_lb_round8; both layouts): a producer warp takes tiles in ticket order and streams them into a ring of shared-memory
// stages with bulk copies (TMA) that complete on mbarriers; other warps rank
// each tile's digits stably, publish the tile's per-digit counts, reorder the
// tile by digit in shared memory, resolve the global per-digit offsets by
// look-back, and store each digit run into its output blocks (Radsort) or
// contiguously (out of place).  Look-back words live in a ring of R tiles x
// sigma 64-bit words: (tag << 32) | value, the tag naming the round and the
// tile, the value the tile's count or 0x80000000 | inclusive prefix (n < 2^31).  Tile t
// reuses the slot of tile t - R only after every tile up to t - R + 1 has
// finished its look-back (per-slot done tags that the producer checks).  A
// reader that finds a slot already reused starts its look-back over: tile
// t - R + 1 is inclusive by then, so the new walk stops above the reused slot.
#include <type_traits>

#include "rs_common.cuh"
#include "rs_kernels.cuh"

namespace rs {

unsigned take_status_oop() { return take_status_word(); }

namespace {

constexpr uint32_t LB_INCL = 0x80000000u;
constexpr uint32_t PI_NONE = 0xFFFFFFFFu;
constexpr uint32_t TILE_END = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t *p)
{
    return *reinterpret_cast<const volatile uint32_t *>(p);
}
__device__ __forceinline__ void st_volatile(uint32_t *p, uint32_t v)
{
    *reinterpret_cast<volatile uint32_t *>(p) = v;
}
__device__ __forceinline__ unsigned long long ld_volatile64(const unsigned long long *p)
{
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}
__device__ __forceinline__ void st_volatile64(unsigned long long *p, unsigned long long v)
{
    *reinterpret_cast<volatile unsigned long long *>(p) = v;
}
__device__ __forceinline__ unsigned long long lbw(uint32_t tag, uint32_t v)
{
    return (static_cast<unsigned long long>(tag) << 32) | v;
}

// ---------------------------------------------------------------- digit histograms
// 8-bit digits: counts of four digit positions r0 .. r0+3 with one counter
// column per lane (counter (r, d) of lane l at word (r*256 + d)*32 + l), so
// the 32 atomics of a warp instruction fall in 32 different banks whatever
// the digits.  One CTA of 1024 threads per SM, 128 KB of counters.  FLT: float32
// keys, counted as ordered integers (a run-time switch made the counts of all
// keys 0.25 -> 0.33 ms at 2^28).
template <typename KT, bool FLT = false>
__global__ void __launch_bounds__(1024) k_digit_hist_lanes(const KT *keys, uint32_t n, int r0, uint32_t *hist)
{
    constexpr int NTD = 8 * int(sizeof(KT)) / 8;
    constexpr int G = 4; // digit positions per pass
    constexpr int V = 16 / sizeof(KT);
    extern __shared__ uint32_t sh[]; // G * 256 * 32
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < G * 256 * 32; i += blockDim.x)
        sh[i] = 0;
    __syncthreads();
    const int npos = min(G, NTD - r0);
    auto put = [&](KT k) {
        if constexpr (FLT)
            k = float_to_ordered(k);
#pragma unroll
        for (int r = 0; r < G; ++r)
            if (r < npos)
                atomicAdd(&sh[(r * 256 + digit_of(k, uint32_t((r0 + r) * 8), 255u)) * 32 + lane], 1u);
    };
    const size_t stride = size_t(gridDim.x) * blockDim.x;
    const size_t first = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const bool vec = (reinterpret_cast<uintptr_t>(keys) & 15u) == 0;
    const size_t nv = vec ? n / V : 0;
    const uint4 *kv = reinterpret_cast<const uint4 *>(keys);
    constexpr int U = 4;
    for (size_t i = first; i < nv; i += U * stride) {
        uint4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < nv)
                v[u] = kv[i + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < nv) {
                KT k[V];
                memcpy(k, &v[u], 16);
#pragma unroll
                for (int q = 0; q < V; ++q)
                    put(k[q]);
            }
    }
    for (size_t i = nv * V + first; i < n; i += stride)
        put(keys[i]);
    __syncthreads();
    // per (position, digit): the sum of the 32 lane columns
    for (int i = threadIdx.x; i < npos * 256; i += blockDim.x) {
        const uint32_t *row = sh + size_t(i) * 32;
        uint32_t sum = 0;
#pragma unroll
        for (int l = 0; l < 32; ++l)
            sum += row[(l + i) & 31]; // rotated start: consecutive threads, different banks
        if (sum)
            atomicAdd(&hist[(r0 + i / 256) * 256 + (i % 256)], sum);
    }
}

// 11-bit digits one by one: counts of all passes (at most 64 buckets each) in one read,
// in counter columns per lane too: 48 or 96 KB of counters.
template <typename KT>
__global__ void __launch_bounds__(1024) k_pass_hist_lanes(const KT *keys, uint32_t n, uint32_t *hist)
{
    constexpr int NP = digit_passes(int(sizeof(KT)), 11, false), B = 64, U = 4;
    extern __shared__ uint32_t sh[]; // NP * B * 32
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < NP * B * 32; i += blockDim.x)
        sh[i] = 0;
    __syncthreads();
    const size_t stride = size_t(gridDim.x) * blockDim.x;
    for (size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += U * stride) {
        KT k[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < n)
                k[u] = keys[i + u * stride];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i + u * stride < n)
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    const DigitPass dp = digit_pass(int(sizeof(KT)), 11, false, q);
                    atomicAdd(&sh[(q * B + digit_of(k[u], dp.shift, dp.mask())) * 32 + lane], 1u);
                }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < NP * B; i += blockDim.x) {
        const uint32_t *row = sh + size_t(i) * 32;
        uint32_t sum = 0;
#pragma unroll
        for (int l = 0; l < 32; ++l)
            sum += row[(l + i) & 31]; // rotated start: consecutive threads, different banks
        if (sum)
            atomicAdd(&hist[(i / B) * 256 + i % B], sum);
    }
}

// Launches the bucket counts of every pass, by bytes or (11-bit digits one by
// one) by half digits.
static cudaError_t launch_digit_hist(const void *keys, uint32_t n, int kb, bool bytes, bool flt, uint32_t *hist,
                                     cudaStream_t st)
{
    using u64 = unsigned long long;
    constexpr int LSM = 4 * 256 * 32 * 4;
    constexpr int P4 = digit_passes(4, 11, false) * 64 * 32 * 4, P8 = digit_passes(8, 11, false) * 64 * 32 * 4;
    static DeviceOnce attr;
    const cudaError_t ea = attr.run([] {
        cudaError_t e = cudaFuncSetAttribute(k_digit_hist_lanes<uint32_t>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, LSM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_digit_hist_lanes<uint32_t, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     LSM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_digit_hist_lanes<u64>, cudaFuncAttributeMaxDynamicSharedMemorySize, LSM);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_pass_hist_lanes<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, P4);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_pass_hist_lanes<u64>, cudaFuncAttributeMaxDynamicSharedMemorySize, P8);
        return e;
    });
    if (ea != cudaSuccess)
        return ea;
    const int grid = num_sms();
    g_launches += 1;
    if (bytes) {
        if (kb == 4 && flt) {
            k_digit_hist_lanes<uint32_t, true><<<grid, 1024, LSM, st>>>(static_cast<const uint32_t *>(keys), n, 0, hist);
        } else if (kb == 4) {
            k_digit_hist_lanes<uint32_t><<<grid, 1024, LSM, st>>>(static_cast<const uint32_t *>(keys), n, 0, hist);
        } else {
            for (int r0 = 0; r0 < 8; r0 += 4)
                k_digit_hist_lanes<u64><<<grid, 1024, LSM, st>>>(static_cast<const u64 *>(keys), n, r0, hist);
            g_launches += 1;
        }
    } else if (kb == 4) {
        k_pass_hist_lanes<uint32_t><<<2 * grid, 1024, P4, st>>>(static_cast<const uint32_t *>(keys), n, hist);
    } else {
        k_pass_hist_lanes<u64><<<grid, 1024, P8, st>>>(static_cast<const u64 *>(keys), n, hist);
    }
    return cudaGetLastError();
}

// Exclusive scan over an N-element array by NT threads (each thread a run of
// IPT consecutive elements); returns the total.  t: the caller's index among
// the NT threads (whole warps: thread t is lane t % 32 of the group's warp
// t / 32), bar: a barrier over exactly those threads.  tmp: NT/32+1 words.
// Ends with a barrier.
template <int N, int NT, typename F>
__device__ __forceinline__ uint32_t block_scan(uint32_t *a, uint32_t *tmp, F &&bar, int t)
{
    constexpr int NWARP = NT / 32;
    constexpr int IPT = (N + NT - 1) / NT;
    const int lane = t & 31, w = t >> 5;
    uint32_t v[IPT], s = 0;
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const int idx = t * IPT + i;
        v[i] = idx < N ? a[idx] : 0;
        s += v[i];
    }
    const uint32_t inc = warp_incl_scan(s);
    if (lane == 31)
        tmp[w] = inc;
    bar();
    if (w == 0) {
        const uint32_t x = lane < NWARP ? tmp[lane] : 0;
        const uint32_t sx = warp_incl_scan(x);
        if (lane < NWARP)
            tmp[lane] = sx - x;
        if (lane == 31)
            tmp[NWARP] = sx;
    }
    bar();
    uint32_t e = inc - s + tmp[w];
#pragma unroll
    for (int i = 0; i < IPT; ++i) {
        const int idx = t * IPT + i;
        if (idx < N)
            a[idx] = e;
        e += v[i];
    }
    const uint32_t tot = tmp[NWARP];
    bar();
    return tot;
}

// Bucket offsets of every pass of the out-of-place sort: O[r][c] exclusive over
// buckets, O[r][256] = n (one block per pass).
__global__ void __launch_bounds__(256) k_offsets(const uint32_t *hist, uint32_t *off, uint32_t n)
{
    constexpr int SIGMA = 256;
    __shared__ uint32_t s_a[SIGMA], s_tmp[16];
    const int r = blockIdx.x;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x)
        s_a[c] = hist[r * SIGMA + c];
    __syncthreads();
    block_scan<SIGMA, SIGMA>(s_a, s_tmp, [] { __syncthreads(); }, threadIdx.x);
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x)
        off[r * (SIGMA + 1) + c] = s_a[c];
    if (threadIdx.x == 0)
        off[r * (SIGMA + 1) + SIGMA] = n;
}

// ---------------------------------------------------------------- grid layout: setup, tables
// Tables of one round, in words of Bufs::tab (GRID_TAB_WORDS a round): bucket
// starts O (sigma + 1), each bucket's range of non-shared blocks [ns0, ns1),
// the free-list index of its first one, the shared blocks (those with a bucket
// start strictly inside) in order, and a header.
enum { TAB_SKIP = 0, TAB_TAKEN = 1, TAB_NS = 2 }; // identity round; free-list entries taken before it; shared blocks
struct GridTab {
    static constexpr int SIGMA = 256, O = 0, NS0 = SIGMA + 1, NS1 = NS0 + SIGMA, FREE = NS1 + SIGMA, SHARED = FREE + SIGMA,
                         HDR = SHARED + SIGMA, WORDS = HDR + 3;
};

// The tables of rounds r0 .. r0 + nr - 1 from the digit counts alone, one CTA
// of 1024 threads each; the other CTAs (setup) write the first map,
// pi = [scratch 0 .. H) ++ [A's blocks] ++ [scratch block H: the input tail],
// and copy that tail.  A digit with one non-empty bucket leaves the sequence
// unchanged: its round is skipped.
template <typename KT>
__global__ void __launch_bounds__(1024)
    k_grid_tables(const uint32_t *hist, uint32_t *tab, uint32_t r0, uint32_t nr, uint32_t n, uint32_t lb, uint32_t H,
                  uint32_t nA, uint32_t npi, const KT *Ak, const uint32_t *Av, KT *Tk, uint32_t *Tv, uint32_t *pi,
                  uint2 *P, uint32_t *state)
{
    using T = GridTab;
    constexpr int SIGMA = T::SIGMA;
    const uint32_t b = 1u << lb;
    if (blockIdx.x >= nr) { // setup (Alg. 4)
        const uint32_t id = (blockIdx.x - nr) * blockDim.x + threadIdx.x, step = (gridDim.x - nr) * blockDim.x;
        const uint32_t nT = H + 1, tail = n - nA * b;
        for (uint32_t i = id; i < npi; i += step)
            pi[i] = i < H ? i : (i < H + nA ? nT + (i - H) : H);
        for (uint32_t j = id; j < tail; j += step) {
            Tk[size_t(H) * b + j] = Ak[size_t(nA) * b + j];
            if (Av)
                Tv[size_t(H) * b + j] = Av[size_t(nA) * b + j];
        }
        if (id == 0) {
            P[0] = make_uint2(H + nA, tail);
            state[ST_F] = H + nA + 1;
            state[ST_NP] = 1;
            state[ST_FPREV] = H + nA + 1;
            state[ST_LOFFTOT] = 0;
        }
        return;
    }
    // s_a: scan buffer; s_list: bucket of the k-th bucket start strictly
    // inside a block, later the k-th shared block
    __shared__ uint32_t s_O[SIGMA + 1], s_cnt[SIGMA], s_a[SIGMA], s_list[SIGMA], s_tmp[40];
    const uint32_t *hist_r = hist + size_t(r0 + blockIdx.x) * SIGMA;
    uint32_t *t = tab + size_t(r0 + blockIdx.x) * T::WORDS;
    auto bar = [] { __syncthreads(); };
    bool one = false;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x) {
        const uint32_t v = hist_r[c];
        s_cnt[c] = v;
        s_O[c] = v;
        one |= v == n;
    }
    if (__syncthreads_or(one)) {
        if (threadIdx.x == 0)
            t[T::HDR + TAB_SKIP] = 1;
        return;
    }
    block_scan<SIGMA, 1024>(s_O, s_tmp, bar, threadIdx.x);
    if (threadIdx.x == 0)
        s_O[SIGMA] = n;
    // bucket starts strictly inside a block, in order
    auto inner = [&](int c) { return s_cnt[c] > 0 && (s_O[c] & (b - 1)) != 0; };
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x)
        s_a[c] = inner(c) ? 1u : 0u;
    __syncthreads();
    block_scan<SIGMA, 1024>(s_a, s_tmp, bar, threadIdx.x);
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x)
        if (inner(c))
            s_list[s_a[c]] = static_cast<uint32_t>(c);
    __syncthreads();
    // the first start inside each block makes it a shared block
    uint32_t fl[(SIGMA + 1023) / 1024];
    int q = 0;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x, ++q) {
        bool first = false;
        if (inner(c)) {
            const uint32_t r = s_a[c];
            first = r == 0 || (s_O[s_list[r - 1]] >> lb) != (s_O[c] >> lb);
        }
        fl[q] = first ? 1u : 0u;
    }
    __syncthreads();
    q = 0;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x, ++q)
        s_a[c] = fl[q];
    __syncthreads();
    const uint32_t nS = block_scan<SIGMA, 1024>(s_a, s_tmp, bar, threadIdx.x);
    q = 0;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x, ++q)
        if (fl[q])
            s_list[s_a[c]] = s_O[c] >> lb;
    __syncthreads();
    auto shared = [&](uint32_t j) -> bool { // is block j shared?
        uint32_t lo = 0, hi = nS;
        while (lo < hi) {
            const uint32_t m = (lo + hi) >> 1;
            if (s_list[m] < j)
                lo = m + 1;
            else
                hi = m;
        }
        return lo < nS && s_list[lo] == j;
    };
    uint32_t ahead[(SIGMA + 1023) / 1024];
    q = 0;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x, ++q) {
        const uint32_t O = s_O[c], cn = s_cnt[c];
        uint32_t ns0, ns1;
        if (cn > 0) {
            const uint32_t jf = O >> lb, jl = (O + cn - 1) >> lb;
            ns0 = jf + (shared(jf) ? 1u : 0u);
            ns1 = jl + 1 - (shared(jl) ? 1u : 0u);
            if (ns1 < ns0)
                ns1 = ns0;
        } else {
            ns0 = ns1 = (O + b - 1) >> lb;
        }
        t[T::O + c] = O;
        t[T::NS0 + c] = ns0;
        t[T::NS1 + c] = ns1;
        if (uint32_t(c) < nS)
            t[T::SHARED + c] = s_list[c];
        ahead[q] = min(GRID_AHEAD, ns1 - ns0);
    }
    __syncthreads();
    // the first GRID_AHEAD non-shared blocks of each bucket: entries nS .. nP-1
    q = 0;
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x, ++q)
        s_a[c] = ahead[q];
    __syncthreads();
    const uint32_t nF = block_scan<SIGMA, 1024>(s_a, s_tmp, bar, threadIdx.x);
    for (int c = threadIdx.x; c < SIGMA; c += blockDim.x)
        t[T::FREE + c] = nS + s_a[c];
    if (threadIdx.x == 0) {
        t[T::O + SIGMA] = n;
        t[T::HDR + TAB_SKIP] = 0;
        t[T::HDR + TAB_TAKEN] = nS + nF;
        t[T::HDR + TAB_NS] = nS;
    }
}

// pi' before a round, an entry per thread: the next head start (the H
// free-list entries after the last one taken), the blocks taken before the
// round (shared block k takes entry k, then the first non-shared blocks of
// each bucket theirs), the empty tail block when b divides n, and unset
// entries for the blocks that the round takes.  An identity round copies pi.
// Latency bounds it: one CTA that made the round's tables and wrote the map
// took 10-12 us a round (and a memset before it past 65536 blocks); the tables
// of all rounds in one launch at setup and this kernel take 8 + 4 x 6 us of a
// sort of 2^20 where that took 45.
__global__ void __launch_bounds__(256)
    k_grid_fill(const uint32_t *tab, uint32_t n, uint32_t lb, uint32_t H, uint32_t nA, uint32_t npi,
                const uint32_t *pi, uint32_t *pin)
{
    using T = GridTab;
    constexpr int SIGMA = T::SIGMA;
    __shared__ uint32_t s_O[SIGMA + 1], s_list[SIGMA];
    const uint32_t skip = tab[T::HDR + TAB_SKIP], nS = skip ? 0u : tab[T::HDR + TAB_NS];
    if (!skip) {
        for (int c = threadIdx.x; c <= SIGMA; c += blockDim.x)
            s_O[c] = tab[T::O + c];
        for (uint32_t k = threadIdx.x; k < nS; k += blockDim.x)
            s_list[k] = tab[T::SHARED + k];
    }
    __syncthreads();
    const uint32_t b = 1u << lb, NB = (n + b - 1) >> lb;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < npi; i += gridDim.x * blockDim.x) {
        // (the round reads free-list entries 0 .. H + nA only; blocks past
        // them, free blocks left behind when the sequence was cut short,
        // Alg. 8, keep their map entries)
        uint32_t from = i; // pi entry that pi'[i] is
        if (!skip && i < H) {
            from = NB + i;
        } else if (!skip && i <= H + nA) {
            const uint32_t j = i - H;
            if (j >= NB) {
                from = NB + H;
            } else {
                const uint32_t p = j << lb;
                uint32_t lo = 0, hi = SIGMA; // the bucket of position p: the last with O <= p
                while (hi - lo > 1) {
                    const uint32_t m = (lo + hi) >> 1;
                    if (s_O[m] <= p)
                        lo = m;
                    else
                        hi = m;
                }
                const uint32_t next = s_O[lo + 1];
                if (next < n && next - p < b) { // shared
                    uint32_t l = 0, h = nS;
                    while (l < h) {
                        const uint32_t m = (l + h) >> 1;
                        if (s_list[m] < j)
                            l = m + 1;
                        else
                            h = m;
                    }
                    from = l;
                } else {
                    const uint32_t ns0 = tab[T::NS0 + lo];
                    from = j - ns0 < GRID_AHEAD ? tab[T::FREE + lo] + (j - ns0) : PI_NONE;
                }
            }
        }
        pin[i] = from == PI_NONE ? PI_NONE : pi[from];
    }
}

// ---------------------------------------------------------------- round kernel
template <typename KT> struct LbArgs {
    const KT *ik;           // out of place: source
    const uint32_t *iv;
    KT *ok;                 // out of place: destination
    uint32_t *ov;
    KT *Ak;                 // Radsort: block storage (A's blocks after nT scratch blocks)
    uint32_t *Av;
    KT *Tk;
    uint32_t *Tv;
    const uint32_t *pi;     // Radsort: current block map (= the free list)
    uint32_t *pin;          // Radsort: next block map
    const uint32_t *tab;    // O[sigma+1] (+ Radsort: ns0, ns1)
    unsigned long long *ring; // R x sigma look-back words (tags below tagbase)
    uint32_t *done;         // R done tags
    uint32_t *ticket;       // zeroed
    uint32_t rmask;         // R - 1 (R a power of two)
    uint32_t tagbase;       // tag of tile t: tagbase + t (grows with the round)
    const uint32_t *hdr;    // Radsort: the tables' header
    uint32_t n, ntiles, H, nT, npi, lb;
    uint32_t shift, mask;   // the pass's digit: key >> shift & mask, at most 255
    // FLT kernels: float32 keys, made ordered (1) or floats again (2) by this
    // pass.  A transform of its own reads and writes every key: 0.135 ms before
    // and after a sort of 2^26 (2.56 ms in all; 2.33 without them)
    uint32_t flt;
};

// Exclusive prefix of bucket c before tile t: sum of the counts of the tiles
// back to the nearest inclusive prefix, LBW words in flight per step.
template <int SIGMA, int LBW = 8>
__device__ __forceinline__ uint32_t look_back(const unsigned long long *ring, uint32_t rmask,
                                              uint32_t tagbase, uint32_t t, int c)
{
    uint32_t excl = 0;
    int x = static_cast<int>(t) - 1;
    unsigned spins = 0;
    while (x >= 0) {
        unsigned long long v[LBW];
#pragma unroll
        for (int k = 0; k < LBW; ++k)
            v[k] = x - k >= 0 ? ld_volatile64(ring + size_t((x - k) & rmask) * SIGMA + c)
                              : lbw(0xFFFFFFFFu, LB_INCL);
        int k = 0;
        for (; k < LBW; ++k) {
            const int y = x - k;
            const uint32_t want = y >= 0 ? tagbase + uint32_t(y) : 0xFFFFFFFFu;
            const uint32_t tag = static_cast<uint32_t>(v[k] >> 32), s = static_cast<uint32_t>(v[k]);
            if (tag != want) {
                if (tag > want) {
                    // the slot was reused, so tile y + 1 has finished and is
                    // inclusive by now: start over from tile t - 1
                    excl = 0;
                    x = static_cast<int>(t) - 1 + k; // x - k below = t - 1
                }
                break; // tile y has not published yet (or restart)
            }
            if (s & LB_INCL)
                return excl + (s & ~LB_INCL);
            excl += s;
        }
        x -= k;
        if (k < LBW) {
            if (++spins > SPIN_LIMIT || ((spins & 1023u) == 0 && wait_failed())) {
                set_status(ST_TIMEOUT);
                return excl;
            }
            // wait for that tile's word alone: reloading the whole window
            // loads the L2 with polls (round kernel at 2^28: 1.58 ms, so 1.53)
            while (x >= 0) {
                const unsigned long long w = ld_volatile64(ring + size_t(x & rmask) * SIGMA + c);
                if (static_cast<uint32_t>(w >> 32) >= tagbase + uint32_t(x))
                    break;
                if (++spins > SPIN_LIMIT || ((spins & 1023u) == 0 && wait_failed())) {
                    set_status(ST_TIMEOUT);
                    return excl;
                }
                __nanosleep(64);
            }
        }
    }
    return excl;
}

__device__ __forceinline__ uint32_t wait_pi(const uint32_t *p)
{
    for (unsigned it = 0; it < SPIN_LIMIT; ++it) {
        const uint32_t v = ld_volatile(p);
        if (v != PI_NONE)
            return v;
        if ((it & 1023u) == 1023u && wait_failed())
            return PI_NONE;
        __nanosleep(64);
    }
    set_status(ST_TIMEOUT);
    return PI_NONE;
}

// One CTA per SM: NW ranking warps, 8 look-back warps and a producer warp, on
// tiles of TILE elements in two shared-memory stages.  What bounds it is
// shared memory (the random-digit accesses of the ranking and the reorder,
// each 3.4 wavefronts a row of 32 elements), 75% busy, then instruction issue,
// 48%; DRAM is at 36% of its peak.  Hence
//  * the ranking works on half-warps.  Each half-warp ranks its own run of
//    TILE / (2 NW) elements, 16 a row, with one word per digit: the count so
//    far in the high half, the lanes of this row in the low half.  A row is
//    one atomicOr, one read and one write by the last lane of each digit
//    group; a word per warp needs mask and count apart (two reads, two
//    writes).  Ranking a tile of 10240: 5600 -> 3450 cycles.
//  * the look-back and the block lists (5-6 L2 round trips, 4.6 us a tile) run
//    on their own warps, one thread per bucket.  The ranking warps rank and
//    count tile k before they store tile k - 1, so tile k's look-back has that
//    store, the reorder of tile k and the ranking of tile k + 1 to complete
//    in, and no one waits for it.
//  * no barrier ends a tile: a warp that has stored and reordered its part
//    ranks the next tile.
// Measured (a round, uniform keys, ms; before: 16 ranking warps that did all
// of it in turn, per-warp masks and counts): 2^28 u32 + u32 1.79 -> 1.46, u32
// alone 1.48 -> 0.92; 2^27 u64 + u32 1.26 -> 1.06, u64 alone 0.88 -> 0.69;
// 2^26 u32 + u32 Zipf 0.83 -> 0.62.  The look-back walks over 64-bit words, 8
// in flight; smaller words with flags, or groups of tiles with a prefix each,
// read less but need two dependent round trips where the walk needs one, and
// were slower (1.9 to 3 ms at 2^28 u32 + u32).
template <typename KT, bool HASV, int TILE, int NW, bool OOP> struct Lb8Cfg {
    static constexpr int SIGMA = 256, STAGES = 2;
    static constexpr int NT = NW * 32;             // ranking threads
    static constexpr int NA = SIGMA;               // look-back threads, one per bucket
    static constexpr int THREADS = NT + NA + 128;  // + the producer's warpgroup
    static constexpr int NPW = OOP ? 1 : 4;        // its warps that work
    static constexpr int SROWS = 2 * NW;           // half-warps
    static constexpr int R = TILE / SROWS;         // elements ranked per half-warp
    static constexpr int ITEMS = R / 16;           // elements per ranking thread
    static_assert(TILE % (NW * 64) == 0 && R % 16 == 0 && ITEMS % 2 == 0, "whole rows, an even number");
    static constexpr int PARTS = NT / SIGMA;       // threads per bucket in the column pass
    static constexpr int RPT = SROWS / PARTS;      // rows each of them sums
    static_assert(PARTS * SIGMA == NT && (PARTS == 1 || PARTS == 2), "one or two threads per bucket");
    static constexpr int MAXM = TILE / 64;         // blocks per tile (b >= 64)
    static constexpr bool PAIR = HASV && sizeof(KT) == 4;
    // touched blocks per tile: at most TILE/b + 2 per bucket with elements
    static constexpr int LIST = MAXM + 2 * SIGMA + 2;
    static constexpr size_t al(size_t x) { return (x + 127) & ~size_t(127); }
    // 16 bytes of slack per array: the lead of a misaligned source (out of
    // place).  The values start 64 bytes past a multiple of 128, so that one
    // half-warp reading keys and the other values meet in no bank
    static constexpr size_t KBYTES = al(size_t(TILE) * sizeof(KT) + 16 + 64) - 64;
    static constexpr size_t STAGE = al(KBYTES + (HASV ? size_t(TILE) * 4 + 16 : 0));
    static constexpr size_t o_tab = STAGES * STAGE;                  // SROWS x SIGMA words
    // what the look-back warps read or write of a tile while the ranking
    // warps work on the next one is there twice (even and odd tiles)
    static constexpr size_t o_part = o_tab + size_t(SROWS) * SIGMA * 4; // 2 x PARTS x SIGMA
    static constexpr size_t o_bst = o_part + 2 * size_t(PARTS) * SIGMA * 4; // 2 x SIGMA
    static constexpr size_t o_tot = o_bst + 2 * size_t(SIGMA) * 4;   // 8 x 16 bytes, then 8 words
    static constexpr size_t QD = size_t(SIGMA) * 16;                 // run descriptors
    static constexpr size_t LISTB = OOP ? 0 : al(size_t(LIST) * 8);
    static constexpr size_t o_qd = o_tot + 256;                      // 2 x QD
    static constexpr size_t o_qlo = o_qd + 2 * QD;                   // 2 x SIGMA
    static constexpr size_t o_list = o_qlo + 2 * size_t(SIGMA) * 4;  // 2 x LISTB
    static constexpr size_t o_tabs = o_list + 2 * LISTB;             // O, ns0, ns1
    static constexpr size_t o_misc = o_tabs + al((3 * size_t(SIGMA) + 4) * 4);
    static constexpr size_t o_meta = o_misc + 64;
    static constexpr size_t o_bar = o_meta + STAGES * 16;
    static constexpr size_t SMEM = al(o_bar + STAGES * 8);
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
    static constexpr int MINB = NW <= 8 && 2 * (SMEM + 1024) <= 228 * 1024 ? 2 : 1; // CTAs per SM
    // registers a thread: a CTA is launched with 72 (896 threads), 48 (two of
    // 640) or 96 (one of 640) and deals them out anew
    static constexpr int MAIN_REGS = NW == 16 ? 88 : MINB == 2 ? 64 : 120;
    static constexpr int AUX_REGS = NW == 16 ? 56 : MINB == 2 ? 40 : 72;
    static constexpr int PROD_REGS = NW == 16 ? 40 : MINB == 2 ? 32 : 72;
};

// Moves registers between the warps of a CTA (all four warps of a warpgroup
// execute it; the shares add up to what the CTA was launched with).
template <int N> __device__ __forceinline__ void reg_dec()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N> __device__ __forceinline__ void reg_inc()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// named barriers of k_lb_round8
enum { LB8_MAIN = 1, LB8_AUX = 2, LB8_CNT = 3, LB8_SCAN = 4, LB8_LIST = 5, LB8_FREE = 6, LB8_PROD = 7 };

// Several arrays sorted out of place in one launch per round (GRP): their
// tiles follow one another, array by array, and the first tile of each has the
// prefix 0, where its other tiles' look-back ends.
struct LbGroup {
    uint32_t narr;
    uint32_t tile0[SEG_GROUP];                 // first tile
    uint32_t len[SEG_GROUP];
    unsigned long long in[SEG_GROUP], out[SEG_GROUP]; // first element in ik / iv and in ok / ov
};
struct LbNoGroup {};

template <typename KT, bool HASV, int TILE, int NW, bool OOP, bool GRP = false, bool FLT = false>
__global__ void __launch_bounds__(Lb8Cfg<KT, HASV, TILE, NW, OOP>::THREADS, Lb8Cfg<KT, HASV, TILE, NW, OOP>::MINB)
    k_lb_round8(LbArgs<KT> a, const __grid_constant__ std::conditional_t<GRP, LbGroup, LbNoGroup> grp)
{
    static_assert(OOP || !GRP, "groups go out of place");
    using C = Lb8Cfg<KT, HASV, TILE, NW, OOP>;
    constexpr int SIGMA = C::SIGMA, NT = C::NT, ITEMS = C::ITEMS;
    extern __shared__ __align__(128) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (!OOP && a.hdr[TAB_SKIP])
        return; // the digit is constant: the round is the identity
    uint32_t *tab = reinterpret_cast<uint32_t *>(sm + C::o_tab);
    uint32_t *part2 = reinterpret_cast<uint32_t *>(sm + C::o_part);
    uint32_t *bst2 = reinterpret_cast<uint32_t *>(sm + C::o_bst);
    uint4 *tot4 = reinterpret_cast<uint4 *>(sm + C::o_tot);
    uint32_t *wsum = reinterpret_cast<uint32_t *>(sm + C::o_tot + 128);
    uint32_t *sO = reinterpret_cast<uint32_t *>(sm + C::o_tabs); // sigma + 1 entries
    uint32_t *misc = reinterpret_cast<uint32_t *>(sm + C::o_misc); // [0..1]: list entries of the tile
    uint32_t *meta = reinterpret_cast<uint32_t *>(sm + C::o_meta);
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + C::o_bar);
    const uint32_t b = 1u << a.lb;

    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(&full[s], C::NPW);
            meta[s * 4] = TILE_END;
        }
        misc[0] = misc[1] = 0;
        fence_mbar_init();
    }
    if constexpr (!GRP)
        for (int c = tid; c < (OOP ? SIGMA + 1 : 3 * SIGMA + 1); c += C::THREADS)
            sO[c] = a.tab[c];
    for (int i = tid; i < C::SROWS * SIGMA; i += C::THREADS)
        tab[i] = 0u;
    __syncthreads();

    if (warp >= NW + SIGMA / 32) {
        // ============================================================ producer
        reg_dec<C::PROD_REGS>();
        const int pw = warp - (NW + SIGMA / 32); // the first draws tickets, all copy (Radsort: a block each lane)
        if (pw >= C::NPW)
            return;
        auto kaddr = [&](uint32_t blk) -> KT * {
            return blk < a.nT ? a.Tk + (size_t(blk) << a.lb) : a.Ak + (size_t(blk - a.nT) << a.lb);
        };
        auto vaddr = [&](uint32_t blk) -> uint32_t * {
            return blk < a.nT ? a.Tv + (size_t(blk) << a.lb) : a.Av + (size_t(blk - a.nT) << a.lb);
        };
        // fill fk (this CTA's tile fk) goes to stage fk % 2
        uint32_t ft = 0, fphys = 0, wm = 0; // drawn ticket; its block bi; tiles below wm have looked back
        const uint32_t bi = uint32_t(lane * C::NPW + pw);
        auto draw = [&](int fk) {
            uint32_t t = 0;
            if (pw == 0 && lane == 0)
                t = atomicAdd(a.ticket, 1u);
            ft = __shfl_sync(0xffffffffu, t, 0);
            if constexpr (!OOP) {
                if (pw == 0 && lane == 0)
                    misc[2 + (fk & 1)] = ft;
                named_bar(LB8_PROD, C::NPW * 32);
                ft = misc[2 + (fk & 1)];
                if (ft < a.ntiles) {
                    const uint32_t cnt = min(uint32_t(TILE), a.n - ft * uint32_t(TILE));
                    const uint32_t nb = (cnt + b - 1) >> a.lb;
                    fphys = bi < nb ? a.pi[a.H + ft * (uint32_t(TILE) >> a.lb) + bi] : 0u;
                }
            }
        };
        // the ring slot of tile ft held tile ft - R: wait until every tile up
        // to ft - R + 1 has finished its look-back
        auto ring_free = [&]() {
            if (ft >= a.ntiles || ft <= a.rmask)
                return;
            const uint32_t need = ft - a.rmask + 1; // tiles below it
            unsigned spins = 0;
            while (wm < need) {
                const uint32_t z = wm + lane;
                const bool ok = z >= need || ld_volatile(a.done + (z & a.rmask)) >= a.tagbase + z;
                const unsigned bal = __ballot_sync(0xffffffffu, ok);
                const uint32_t adv = bal == 0xffffffffu ? 32u : uint32_t(__ffs(~bal) - 1);
                wm = min(need, wm + adv);
                if (wm < need && adv < 32u) {
                    if (++spins > SPIN_LIMIT || ((spins & 1023u) == 0 && wait_failed())) {
                        set_status(ST_TIMEOUT);
                        return;
                    }
                    __nanosleep(64);
                }
            }
        };
        auto issue = [&](int fk) {
            const int s = fk % C::STAGES;
            uint32_t *mt = meta + s * 4;
            if (ft >= a.ntiles) { // the end mark
                if (lane == 0) {
                    if (pw == 0)
                        mt[0] = TILE_END;
                    mbar_arrive(&full[s]);
                }
                return;
            }
            unsigned char *st = sm + size_t(s) * C::STAGE;
            KT *stk = reinterpret_cast<KT *>(st);
            uint32_t *stv = reinterpret_cast<uint32_t *>(st + C::KBYTES);
            uint32_t e0 = ft * uint32_t(TILE), n = a.n, arr = 0; // of a group: in array arr
            const KT *ik = a.ik;
            const uint32_t *iv = a.iv;
            if constexpr (GRP) {
                unsigned before = 0; // arrays that begin at or before tile ft
#pragma unroll
                for (uint32_t j = 0; j < SEG_GROUP; j += 32)
                    before += __popc(__ballot_sync(0xffffffffu, j + lane < grp.narr && grp.tile0[j + lane] <= ft));
                arr = before - 1;
                e0 = (ft - grp.tile0[arr]) * uint32_t(TILE);
                n = grp.len[arr];
                ik += grp.in[arr];
                iv += HASV ? grp.in[arr] : 0;
            }
            const uint32_t cnt = min(uint32_t(TILE), n - e0);
            uint32_t leadk = 0, leadv = 0;
            if constexpr (OOP) {
                // the 16-byte-aligned middle by bulk copies, the ragged ends
                // (under 16 bytes each) by plain loads
                const uintptr_t ka = reinterpret_cast<uintptr_t>(ik + e0);
                const uintptr_t kz = ka + uintptr_t(cnt) * sizeof(KT);
                const uintptr_t ka16 = (ka + 15) & ~uintptr_t(15), kz16 = kz & ~uintptr_t(15);
                leadk = static_cast<uint32_t>((ka & 15) / sizeof(KT));
                const bool kmid = ka16 < kz16;
                const uint32_t khead = kmid ? static_cast<uint32_t>((ka16 - ka) / sizeof(KT)) : cnt;
                const uint32_t ktail = kmid ? static_cast<uint32_t>((kz16 - ka) / sizeof(KT)) : cnt;
                uint32_t bytes = kmid ? static_cast<uint32_t>(kz16 - ka16) : 0u;
                uintptr_t va16 = 0, vz16 = 0;
                uint32_t vhead = 0, vtail = 0;
                bool vmid = false;
                if (HASV) {
                    const uintptr_t va = reinterpret_cast<uintptr_t>(iv + e0);
                    const uintptr_t vz = va + uintptr_t(cnt) * 4;
                    va16 = (va + 15) & ~uintptr_t(15);
                    vz16 = vz & ~uintptr_t(15);
                    leadv = static_cast<uint32_t>((va & 15) / 4);
                    vmid = va16 < vz16;
                    vhead = vmid ? static_cast<uint32_t>((va16 - va) / 4) : cnt;
                    vtail = vmid ? static_cast<uint32_t>((vz16 - va) / 4) : cnt;
                    bytes += vmid ? static_cast<uint32_t>(vz16 - va16) : 0u;
                }
                if (lane == 0 && bytes)
                    asm volatile("mbarrier.expect_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])),
                                 "r"(bytes)
                                 : "memory");
                __syncwarp();
                if (lane == 0 && kmid)
                    bulk_g2s(stk + leadk + khead, reinterpret_cast<const void *>(ka16),
                             static_cast<uint32_t>(kz16 - ka16), &full[s]);
                if (HASV && lane == 1 && vmid)
                    bulk_g2s(stv + leadv + vhead, reinterpret_cast<const void *>(va16),
                             static_cast<uint32_t>(vz16 - va16), &full[s]);
                for (uint32_t e = lane; e < khead; e += 32)
                    stk[leadk + e] = ik[e0 + e];
                for (uint32_t e = ktail + lane; e < cnt; e += 32)
                    stk[leadk + e] = ik[e0 + e];
                if (HASV) {
                    for (uint32_t e = lane; e < vhead; e += 32)
                        stv[leadv + e] = iv[e0 + e];
                    for (uint32_t e = vtail + lane; e < cnt; e += 32)
                        stv[leadv + e] = iv[e0 + e];
                }
            } else {
                // blocks ft*M .. of the logical data: block i at stage offset
                // i*b (a block index outside the block store is reported and
                // skipped)
                const uint32_t nb = (cnt + b - 1) >> a.lb;
                const uint32_t i0 = a.H + ft * (uint32_t(TILE) >> a.lb);
                uint32_t tot = 0;
                for (uint32_t base = 0; base < nb; base += 32 * C::NPW) {
                    const uint32_t i = base + bi;
                    uint32_t bytes = 0;
                    if (i < nb && (base ? a.pi[i0 + i] : fphys) < a.npi) {
                        const uint32_t len = min(b, cnt - i * b);
                        bytes = ((len * uint32_t(sizeof(KT)) + 15u) & ~15u) + (HASV ? ((len * 4u + 15u) & ~15u) : 0u);
                    }
                    tot += warp_sum(bytes);
                }
                if (lane == 0 && tot)
                    asm volatile("mbarrier.expect_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])),
                                 "r"(tot)
                                 : "memory");
                __syncwarp();
                for (uint32_t i = bi; i < nb; i += 32 * C::NPW) {
                    const uint32_t len = min(b, cnt - i * b);
                    const uint32_t phys = i == bi ? fphys : a.pi[i0 + i];
                    if (phys >= a.npi) {
                        set_status(ST_INTERNAL);
                        continue;
                    }
                    bulk_g2s(stk + size_t(i) * b, kaddr(phys), (len * uint32_t(sizeof(KT)) + 15u) & ~15u, &full[s]);
                    if (HASV)
                        bulk_g2s(stv + size_t(i) * b, vaddr(phys), (len * 4u + 15u) & ~15u, &full[s]);
                }
            }
            __syncwarp();
            if (pw == 0 && lane == 0) {
                mt[0] = ft;
                mt[1] = cnt;
                mt[2] = leadk | (leadv << 8);
                mt[3] = arr;
            }
            __syncwarp();
            if (lane == 0)
                mbar_arrive(&full[s]); // release: the plain stores above are visible
        };
        // Radsort: the copies of a fill, two a block, are dealt over the four
        // warps, as a warp issues its lanes' copies one after the other, about
        // 0.12 us each: 4.8 us of the 8.4 us a tile with blocks of 512.  A round
        // of 2^20 u32 + u32 23.0 -> 21.3 us, 2^24 110 -> 105 us (blocks of 512),
        // 2^28 unchanged (blocks of 2048).  (2^26 with Zipf keys, whose tiles
        // take unequal times: 2.78 -> 2.82 ms a sort.)
        // The ticket of fill k + 1 is drawn when tile k is counted, not before:
        // every look-back waits for the tiles drawn earlier, and a CTA that
        // drew two tiles in a row at its start held up all between them
        draw(0);
        if (pw == 0)
            ring_free();
        issue(0);
        int k = 0; // fill k is issued
        while (ft < a.ntiles) {
            if (pw == 0)
                named_bar(LB8_CNT, C::NT + C::NA + 32);
            draw(k + 1);
            if (pw == 0)
                ring_free();
            if (k >= 1)
                named_bar(LB8_FREE, NT + C::NPW * 32); // tile k - 1 is stored: the stage of fill k + 1 is free
            issue(++k);
        }
        if (pw != 0)
            return;
        named_bar(LB8_CNT, C::NT + C::NA + 32); // (the end mark's)
        // every issued copy lands before this CTA exits (only after a wait
        // that ran out can one still be in flight)
        if (lane == 0)
            for (int f = k > 0 ? k - 1 : 0; f <= k; ++f)
                mbar_wait(&full[f % C::STAGES], (f / C::STAGES) & 1u);
        return;
    }

    if (warp >= NW) {
        // ============================================================ look-back warps
        reg_dec<C::AUX_REGS>();
        const int c = tid - NT, aw = warp - NW; // this thread's bucket, its warp among the 8
        const uint32_t *ns0 = sO + SIGMA + 1, *ns1 = ns0 + SIGMA;
        uint32_t Oc = GRP ? 0u : sO[c];
        const uint32_t Oe = GRP ? 0u : sO[c + 1];
        const uint32_t n0 = OOP ? 0u : ns0[c], n1 = OOP ? 0u : ns1[c];
        const uint32_t nP = OOP ? 0u : a.hdr[TAB_TAKEN]; // free-list entries taken before the round
        auto kaddr = [&](uint32_t blk) -> KT * {
            return blk < a.nT ? a.Tk + (size_t(blk) << a.lb) : a.Ak + (size_t(blk - a.nT) << a.lb);
        };

        for (uint32_t k = 0;; ++k) { // fill k
            named_bar(LB8_CNT, C::NT + C::NA + 32); // the tile's counts per bucket are in part
            const uint32_t *part = part2 + (k & 1) * C::PARTS * SIGMA, *bst = bst2 + (k & 1) * SIGMA;
            uint4 *qd16 = reinterpret_cast<uint4 *>(sm + C::o_qd + (k & 1) * C::QD);        // Radsort
            uint32_t *qoff = reinterpret_cast<uint32_t *>(sm + C::o_qd + (k & 1) * C::QD);  // out of place
            uint32_t *qlo = reinterpret_cast<uint32_t *>(sm + C::o_qlo) + (k & 1) * SIGMA;
            unsigned long long *list = reinterpret_cast<unsigned long long *>(sm + C::o_list + (k & 1) * C::LISTB);
            const uint32_t t = meta[(k % C::STAGES) * 4];
            if (t == TILE_END)
                break;
            const uint32_t cnt = meta[(k % C::STAGES) * 4 + 1];
            uint32_t t_first = 0, arr = 0; // the array's first tile
            if constexpr (GRP) {
                arr = meta[(k % C::STAGES) * 4 + 3];
                t_first = grp.tile0[arr];
                Oc = __ldg(a.tab + size_t(arr) * (SIGMA + 1) + c);
            }
            // elements past the tile's end were ranked as the largest digit
            uint32_t cn = part[c] + (C::PARTS == 2 ? part[SIGMA + c] : 0u);
            if (uint32_t(c) == a.mask)
                cn -= uint32_t(TILE) - cnt;
            // ---- the count published, the bucket's prefix over the tiles before
            unsigned long long *slot = a.ring + size_t(t & a.rmask) * SIGMA + c;
            st_volatile64(slot, lbw(a.tagbase + t, t == t_first ? (LB_INCL | cn) : cn));
            uint32_t excl = 0;
            if (t > t_first) {
                excl = look_back<SIGMA>(a.ring, a.rmask, a.tagbase, t, c);
                st_volatile64(slot, lbw(a.tagbase + t, LB_INCL | (excl + cn)));
            }
            __syncwarp();
            const uint32_t g = Oc + excl;
            __syncwarp();
            if constexpr (OOP) {
                named_bar(LB8_AUX, C::NA);
                if (c == 0) // this tile reads no more look-back words
                    st_volatile(a.done + (t & a.rmask), a.tagbase + t);
                named_bar(LB8_SCAN, C::NT + C::NA); // bucket starts in the tile
                qoff[c] = g - bst[c];
                if (GRP && c == 0)
                    misc[k & 1] = arr;
            } else {
                // the run lies inside the bucket's output range unless the
                // look-back words were corrupted: then it is reported and its
                // blocks are left alone
                if (g + cn > Oe || g + cn < g) {
                    set_status(ST_INTERNAL);
                    cn = 0;
                }
                // ---- blocks touched, blocks taken here and by earlier tiles
                const uint32_t e = g + cn, j0 = g >> a.lb;
                const uint32_t touched = cn ? ((e - 1) >> a.lb) - j0 + 1 : 0u;
                const uint32_t cs = (g + b - 1) >> a.lb, ce = (e + b - 1) >> a.lb;
                // block j in [n0 + L, n1) is taken by the writer of the first
                // position of block j - L: by earlier tiles for j - L < cs,
                // here for cs <= j - L < ce
                const uint32_t mb = min(cs + GRID_AHEAD, n1), e0 = n0 + GRID_AHEAD;
                const uint32_t before = mb > e0 ? mb - e0 : 0u;
                const uint32_t first = max(cs, n0) + GRID_AHEAD, last = min(ce + GRID_AHEAD, n1);
                const uint32_t take = last > first ? last - first : 0u;
                // the map entry of the first block touched (taken before
                // this tile, if it touches any)
                const uint32_t pf = cn ? ld_volatile(a.pin + a.H + j0) : PI_NONE;
                // (and of the second, where it is not taken here)
                const uint32_t pf2 = touched > 1 && j0 + 1 < first ? ld_volatile(a.pin + a.H + j0 + 1) : PI_NONE;
                const uint32_t it_ = warp_incl_scan(touched), ik = warp_incl_scan(take), sb = warp_sum(before);
                if (lane == 31)
                    tot4[aw] = make_uint4(it_, ik, sb, 0u);
                named_bar(LB8_AUX, C::NA);
                if (c == 0) // this tile reads no more look-back words
                    st_volatile(a.done + (t & a.rmask), a.tagbase + t);
                uint32_t l0 = it_ - touched, ko = ik - take, TT = 0, fbase = nP;
#pragma unroll
                for (int w = 0; w < SIGMA / 32; ++w) {
                    const uint4 x = tot4[w];
                    if (w < aw) {
                        l0 += x.x;
                        ko += x.y;
                    }
                    TT += x.x;
                    fbase += x.z;
                }
                // ---- the physical block of every block this tile touches,
                // and the blocks it takes beyond those.  Those go into the map
                // before this thread waits for any other's: a bucket that
                // fills tile after tile (skewed keys) has each tile continue
                // blocks that the tile just before took, and taking after the
                // wait would chain every tile to its predecessor (1-2 us a
                // tile).  Measured (2^26 keys + index, a sort): Zipf keys 57.8
                // -> 3.7 ms, float32 N(0,1) keys (top digit skewed) 15.8 ->
                // 3.0, uniform keys unchanged
                // free-list entries consumed so far (Lemma 1), within the list
                const uint32_t fcap = min(a.H + (t + 1) * (uint32_t(TILE) >> a.lb), a.npi);
                const uint32_t fi0 = fbase + ko - first; // block j's free-list index - j (mod 2^32)
                for (uint32_t j = first; j < last; ++j) {
                    const uint32_t idx = fi0 + j;
                    if (idx < fcap)
                        a.pin[a.H + j] = __ldg(a.pi + idx);
                    else
                        set_status(ST_INTERNAL); // Lemma 1 would be violated
                }
                __syncwarp();
                named_bar(LB8_SCAN, C::NT + C::NA); // bucket starts in the tile
                // the run's first block is filled in below; an element past
                // it reads its block from the list
                uint4 qd = make_uint4(g - bst[c], 0u, 0u, 0u);
                for (uint32_t i = 0; i < touched; ++i) {
                    const uint32_t j = j0 + i;
                    uint32_t phys;
                    if (j >= first && j < last) { // taken here
                        const uint32_t idx = fi0 + j;
                        phys = idx < fcap ? __ldg(a.pi + idx) : PI_NONE;
                    } else { // taken before the round or by an earlier tile
                        phys = i == 0 ? pf : i == 1 ? pf2 : PI_NONE;
                        if (phys == PI_NONE)
                            phys = wait_pi(a.pin + a.H + j);
                    }
                    if (phys != PI_NONE && phys >= a.npi) {
                        set_status(ST_INTERNAL);
                        phys = PI_NONE;
                    }
                    // one word per entry: the key block pointer, bit 0 set
                    // for a block of A (the value pointer follows from it)
                    const unsigned long long w =
                        phys == PI_NONE ? 0ull
                                        : (reinterpret_cast<unsigned long long>(kaddr(phys)) |
                                           (phys >= a.nT ? 1ull : 0ull));
                    list[l0 + i] = w;
                    if (i == 0 && w) {
                        // the first block as a base for the run's positions:
                        // the key address of position p in it is base + p
                        // elements (bit 1 marks it valid)
                        const unsigned long long base =
                            ((w & ~1ull) - (static_cast<unsigned long long>(j0) << a.lb) * sizeof(KT)) | (w & 1ull) |
                            2ull;
                        qd.y = (j0 + 1) << a.lb;
                        qd.z = static_cast<uint32_t>(base);
                        qd.w = static_cast<uint32_t>(base >> 32);
                    }
                }
                qd16[c] = qd;
                qlo[c] = l0 - j0;
                if (c == 0)
                    misc[k & 1] = TT;
            }
            __syncwarp();
            bar_arrive(LB8_LIST, C::NT + C::NA);
        }
        return;
    }

    // ================================================================ ranking warps
    reg_inc<C::MAIN_REGS>();
    const int h = lane >> 4, l16 = lane & 15;
    uint32_t *row = tab + (2 * warp + h) * SIGMA; // this half-warp's words
    const uint32_t eh = uint32_t((2 * warp + h) * C::R + l16); // its first element in the tile
    auto dig = [&](KT key) -> uint32_t { return digit_of(key, a.shift, a.mask); };

    // Tile k is ranked and counted before tile k - 1 is stored, so that a
    // tile's look-back and block lists have the store before it, its own
    // reorder and the next tile's ranking to complete in.
    uint32_t pcnt = 0; // elements of tile k - 1
    for (uint32_t k = 0;; ++k) { // fill k
        const int s = k % C::STAGES;
        // (a wait that runs out is reported; the tile is then worked through
        // with what is there, so that every barrier is met)
        (void)mbar_wait(&full[s], (k / C::STAGES) & 1u);
        __syncwarp();
        const uint32_t *mt = meta + s * 4;
        const bool end = mt[0] == TILE_END;
        const uint32_t cnt = mt[1], leadk = mt[2] & 0xFFu, leadv = mt[2] >> 8;
        unsigned char *st = sm + size_t(s) * C::STAGE;
        KT *tk = reinterpret_cast<KT *>(st);
        uint32_t *tv = reinterpret_cast<uint32_t *>(st + C::KBYTES);

        KT key[ITEMS];
        uint32_t val[HASV ? ITEMS : 1];
        uint32_t rk[ITEMS / 2]; // ranks within the half-warp, two 16-bit ones each
        if (!end) {
            // ---- 1. this thread's elements into registers
            if constexpr (C::PAIR) {
                // one half-warp reads keys while the other reads values: the two
                // halves' runs start in the same bank
                const uint32_t *p0 = (h ? tv + leadv : tk + leadk) + eh, *p1 = (h ? tk + leadk : tv + leadv) + eh;
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    const uint32_t x = p0[it * 16], y = p1[it * 16];
                    key[it] = h ? y : x;
                    val[it] = h ? x : y;
                }
            } else {
                // (4-byte words: the second half-warp reads the rows of a pair in
                // the other order)
#pragma unroll
                for (int it = 0; it < ITEMS; it += 2) {
                    const KT *pk = tk + leadk + eh + it * 16;
                    if constexpr (sizeof(KT) == 4) {
                        const KT x = pk[h * 16], y = pk[16 - h * 16];
                        key[it] = h ? y : x;
                        key[it + 1] = h ? x : y;
                    } else {
                        key[it] = pk[0];
                        key[it + 1] = pk[16];
                    }
                    if constexpr (HASV) {
                        const uint32_t *pv = tv + leadv + eh + it * 16;
                        const uint32_t x = pv[h * 16], y = pv[16 - h * 16];
                        val[it] = h ? y : x;
                        val[it + 1] = h ? x : y;
                    }
                }
            }
            if constexpr (FLT)
                if (a.flt & 1u) {
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it)
                        key[it] = float_to_ordered(key[it]);
                }
            if (cnt < uint32_t(TILE)) {
                // elements past the end rank as the last ones of the largest digit
#pragma unroll
                for (int it = 0; it < ITEMS; ++it)
                    if (eh + it * 16 >= cnt)
                        key[it] = ~KT(0);
            }
            // ---- stable rank within the half-warp
            rank_half_warp<ITEMS>(row, [&](int it) { return dig(key[it]); }, [](int) { return true; }, rk);
            named_bar(LB8_MAIN, NT);

            // ---- 2. tile counts per bucket, for the look-back warps, and their
            // exclusive scan (bucket starts in the reordered tile); then each
            // half-warp's start per bucket: the ranks are relative to it
            {
                const int c = tid & (SIGMA - 1), p = tid / SIGMA;
                uint32_t *col = tab + p * C::RPT * SIGMA + c;
                uint32_t *part = part2 + (k & 1) * C::PARTS * SIGMA, *bst = bst2 + (k & 1) * SIGMA;
                uint32_t hc[C::RPT / 2], sum = 0;
#pragma unroll
                for (int r = 0; r < C::RPT; r += 2) {
                    const uint32_t x = col[r * SIGMA] >> 16, y = col[(r + 1) * SIGMA] & 0xFFFF0000u;
                    hc[r >> 1] = x | y;
                    sum += x + (y >> 16);
                }
                part[p * SIGMA + c] = sum;
                bar_arrive(LB8_CNT, C::NT + C::NA + 32);
                uint32_t tot = sum, below = 0;
                if constexpr (C::PARTS == 2) {
                    named_bar(LB8_MAIN, NT);
                    const uint32_t o = part[(p ^ 1) * SIGMA + c];
                    tot += o;
                    below = p ? o : 0u;
                }
                const uint32_t inc = warp_incl_scan(tot);
                if (lane == 31 && p == 0)
                    wsum[warp] = inc;
                named_bar(LB8_MAIN, NT);
                uint32_t base = inc - tot;
#pragma unroll
                for (int w = 0; w < SIGMA / 32 - 1; ++w)
                    base += w < (warp & 7) ? wsum[w] : 0u;
                if (p == 0)
                    bst[c] = base;
                uint32_t run = base + below;
#pragma unroll
                for (int r = 0; r < C::RPT; ++r) {
                    col[r * SIGMA] = run;
                    run += (r & 1) ? hc[r >> 1] >> 16 : hc[r >> 1] & 0xFFFFu;
                }
            }
        } else {
            bar_arrive(LB8_CNT, C::NT + C::NA + 32);
        }
        if (k == 0)
            named_bar(LB8_MAIN, NT);
        else
            named_bar(LB8_LIST, C::NT + C::NA); // tile k - 1 is reordered, its run descriptors are there
        if (!end)
            bar_arrive(LB8_SCAN, C::NT + C::NA);

        // ---- 3. store tile k - 1, every bucket run, U elements a thread at a time
        if (k > 0) {
            unsigned char *pst = sm + size_t(s ^ 1) * C::STAGE;
            const KT *pk = reinterpret_cast<const KT *>(pst);
            const uint32_t *pv = reinterpret_cast<const uint32_t *>(pst + C::KBYTES);
            const uint2 *pp = reinterpret_cast<const uint2 *>(pst);
            const unsigned char *qdb = sm + C::o_qd + ((k - 1) & 1) * C::QD;
            const uint4 *qd16 = reinterpret_cast<const uint4 *>(qdb);        // Radsort
            const uint32_t *qoff = reinterpret_cast<const uint32_t *>(qdb);  // out of place
            const uint32_t *qlo = reinterpret_cast<const uint32_t *>(sm + C::o_qlo) + ((k - 1) & 1) * SIGMA;
            const unsigned long long *list =
                reinterpret_cast<const unsigned long long *>(sm + C::o_list + ((k - 1) & 1) * C::LISTB);
            constexpr int SI = TILE / NT, U = SI % 5 == 0 ? 5 : 4;
            static_assert(SI % U == 0, "whole batches");
            const uint32_t TT = OOP ? 0u : misc[(k - 1) & 1];
            KT *ok = a.ok;
            uint32_t *ov = a.ov, n = a.n;
            if constexpr (GRP) {
                const uint32_t arr = misc[(k - 1) & 1];
                ok += grp.out[arr];
                ov += HASV ? grp.out[arr] : 0;
                n = grp.len[arr];
            }
            // byte distance from a key block to its value block, in T and in A
            const long long dvT = reinterpret_cast<const char *>(a.Tv) - reinterpret_cast<const char *>(a.Tk);
            const long long dvA = reinterpret_cast<const char *>(a.Av) - reinterpret_cast<const char *>(a.Ak);
#pragma unroll 1
            for (int k0 = 0; k0 < SI; k0 += U) {
                KT kv[U];
                uint32_t vv[U], idx[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t i = tid + (k0 + u) * NT;
                    if constexpr (C::PAIR) {
                        const uint2 pr = pp[i];
                        kv[u] = pr.x;
                        vv[u] = pr.y;
                    } else {
                        kv[u] = pk[i];
                        vv[u] = HASV ? pv[i] : 0u;
                    }
                }
                if constexpr (OOP) {
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        idx[u] = tid + (k0 + u) * NT + qoff[dig(kv[u])];
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (tid + (k0 + u) * NT < pcnt && idx[u] < n) {
                            ok[idx[u]] = kv[u];
                            if (HASV)
                                ov[idx[u]] = vv[u];
                        }
                } else {
                    // most runs lie in one block, whose base address the run
                    // descriptor holds; the rest read their block from the list,
                    // behind one branch for the warp: a branch per element keeps
                    // the reads of the next ones from overlapping
                    unsigned long long w[U];
                    uint32_t late = 0;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const uint32_t i = tid + (k0 + u) * NT;
                        const uint4 qd = qd16[dig(kv[u])];
                        idx[u] = i + qd.x;
                        w[u] = i < pcnt ? (static_cast<unsigned long long>(qd.w) << 32) | qd.z : 0ull;
                        if (i < pcnt && idx[u] >= qd.y)
                            late |= 1u << u;
                    }
                    if (__any_sync(0xffffffffu, late)) {
#pragma unroll
                        for (int u = 0; u < U; ++u)
                            if ((late >> u) & 1u) {
                                const uint32_t l = (idx[u] >> a.lb) + qlo[dig(kv[u])];
                                w[u] = l < TT ? list[l] : 0ull;
                                idx[u] &= b - 1;
                            }
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (w[u]) {
                            KT *dk = reinterpret_cast<KT *>(w[u] & ~3ull) + idx[u];
                            if constexpr (FLT)
                                *dk = a.flt & 2u ? ordered_to_float(kv[u]) : kv[u];
                            else
                                *dk = kv[u];
                            if (HASV) {
                                uint32_t *dv;
                                if constexpr (sizeof(KT) == 4)
                                    dv = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(dk) +
                                                                      ((w[u] & 1ull) ? dvA : dvT));
                                else
                                    dv = ((w[u] & 1ull) ? a.Av + (dk - a.Ak) : a.Tv + (dk - a.Tk));
                                *dv = vv[u];
                            }
                        }
                }
            }
            // the stage was read and rewritten with generic accesses; it is
            // refilled with bulk copies (async proxy)
            fence_proxy_async_smem();
            bar_arrive(LB8_FREE, NT + C::NPW * 32);
        }
        if (end)
            break;
        pcnt = cnt;

        // ---- 4. reorder the tile by digit, in place in its stage buffer
        // (every element is in registers since the barriers above)
        uint2 *tp = reinterpret_cast<uint2 *>(st); // (key, value) pairs after the reorder
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t pos = row[dig(key[it])] + ((it & 1) ? rk[it >> 1] >> 16 : rk[it >> 1] & 0xFFFFu);
            if (pos >= uint32_t(TILE)) { // only a broken scan gets here
                set_status(ST_INTERNAL);
                continue;
            }
            if constexpr (C::PAIR) {
                tp[pos] = make_uint2(static_cast<uint32_t>(key[it]), val[it]);
            } else {
                tk[pos] = key[it];
                if (HASV)
                    tv[pos] = val[it];
            }
        }
        // this warp's words for the next tile
        __syncwarp();
        {
            uint4 *z = reinterpret_cast<uint4 *>(tab + 2 * warp * SIGMA);
#pragma unroll
            for (int i = 0; i < 2 * SIGMA / 128; ++i)
                z[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
}

// ---------------------------------------------------------------- groups of arrays
// Digit counts (8-bit) of every array of a group: a CTA counts one chunk of
// one array, four digit positions (blockIdx.y: the first four or the last), in
// counter columns per lane as k_digit_hist_lanes does.  hist[array][position].
constexpr uint32_t GRP_CHUNK = 1u << 16;

template <typename KT>
__global__ void __launch_bounds__(1024)
    k_group_hist(const KT *keys, const __grid_constant__ LbGroup grp, uint32_t *hist)
{
    constexpr int NTD = int(sizeof(KT)), G = 4;
    extern __shared__ uint32_t sh[]; // G * 256 * 32
    // the chunk's array: chunks per array follow from its length
    __shared__ uint32_t s_arr, s_chunk;
    if (threadIdx.x == 0) {
        uint32_t b = blockIdx.x, i = 0;
        for (; i < grp.narr; ++i) {
            const uint32_t nch = (grp.len[i] + GRP_CHUNK - 1) / GRP_CHUNK;
            if (b < nch)
                break;
            b -= nch;
        }
        s_arr = i;
        s_chunk = b;
    }
    const int lane = threadIdx.x & 31, r0 = int(blockIdx.y) * G;
    for (int i = threadIdx.x; i < G * 256 * 32; i += blockDim.x)
        sh[i] = 0;
    __syncthreads();
    if (s_arr >= grp.narr)
        return;
    const uint32_t len = grp.len[s_arr], e0 = s_chunk * GRP_CHUNK, e1 = min(e0 + GRP_CHUNK, len);
    const KT *src = keys + grp.in[s_arr];
    constexpr uint32_t U = 8;
    for (uint32_t e = e0 + threadIdx.x; e < e1; e += U * blockDim.x) {
        KT k[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
            if (e + u * blockDim.x < e1)
                k[u] = src[e + u * blockDim.x];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u)
            if (e + u * blockDim.x < e1)
#pragma unroll
                for (int r = 0; r < G; ++r)
                    atomicAdd(&sh[(r * 256 + digit_of(k[u], uint32_t((r0 + r) * 8), 255u)) * 32 + lane], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < G * 256; i += blockDim.x) {
        const uint32_t *rw = sh + size_t(i) * 32;
        uint32_t sum = 0;
#pragma unroll
        for (int l = 0; l < 32; ++l)
            sum += rw[(l + i) & 31]; // rotated start: consecutive threads, different banks
        if (sum)
            atomicAdd(&hist[(size_t(s_arr) * NTD + r0) * 256 + i], sum);
    }
}

// Bucket starts of every array and round: tab[round][array][257].
__global__ void __launch_bounds__(256)
    k_group_offsets(const uint32_t *hist, uint32_t nt, uint32_t narr, const __grid_constant__ LbGroup grp, uint32_t *tab)
{
    __shared__ uint32_t s_a[256], s_tmp[16];
    const uint32_t arr = blockIdx.x % narr, r = blockIdx.x / narr;
    s_a[threadIdx.x] = hist[(size_t(arr) * nt + r) * 256 + threadIdx.x];
    __syncthreads();
    block_scan<256, 256>(s_a, s_tmp, [] { __syncthreads(); }, threadIdx.x);
    uint32_t *t = tab + (size_t(r) * narr + arr) * 257;
    t[threadIdx.x] = s_a[threadIdx.x];
    if (threadIdx.x == 0)
        t[256] = grp.len[arr];
}

// ---------------------------------------------------------------- launch helpers
// The round kernel of a configuration.
template <typename KT, bool HASV, int TILE, int NW, bool OOP> struct LbKernel {
    using C = Lb8Cfg<KT, HASV, TILE, NW, OOP>;
    static constexpr bool FLT = sizeof(KT) == 4 && !OOP; // there is a kernel for float keys
    static void launch(int grid, const LbArgs<KT> &a, cudaStream_t st)
    {
        if (FLT && a.flt)
            k_lb_round8<KT, HASV, TILE, NW, OOP, false, FLT><<<grid, C::THREADS, C::SMEM, st>>>(a, LbNoGroup{});
        else
            k_lb_round8<KT, HASV, TILE, NW, OOP><<<grid, C::THREADS, C::SMEM, st>>>(a, LbNoGroup{});
    }
    // CTAs of a launch over ntiles tiles (-1: the kernel cannot be set up)
    static int ctas(size_t ntiles)
    {
        static DeviceOnce attr; // per template instance
        if (attr.run([] {
                const cudaError_t e = cudaFuncSetAttribute(k_lb_round8<KT, HASV, TILE, NW, OOP>,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
                return e != cudaSuccess || !FLT
                           ? e
                           : cudaFuncSetAttribute(k_lb_round8<KT, HASV, TILE, NW, OOP, false, FLT>,
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
            }) != cudaSuccess)
            return -1;
        size_t grid = size_t(num_sms()) * C::MINB;
        if (grid > ntiles)
            grid = ntiles;
        return grid < 1 ? 1 : static_cast<int>(grid);
    }
};

// Calls f.template operator()<KT, HASV, TILE, NW>() for the configuration.
template <typename F> static cudaError_t lb_dispatch(int kb, bool hasv, F &&f)
{
    using u64 = unsigned long long;
    // The largest tiles that two stages and the tables leave room for
    // (per-tile costs scale with sigma, not with the tile), each a multiple
    // of 2048 so that blocks of up to 2048 elements fit whole.
    if (kb == 4)
        return hasv ? f.template operator()<uint32_t, true, 10240, 16>()
                    : f.template operator()<uint32_t, false, 16384, 16>();
    return hasv ? f.template operator()<u64, true, 6144, 16>() : f.template operator()<u64, false, 10240, 16>();
}

// Radsort rounds with a tile shape: 0 or 1, the configuration above; 2 (8-bit
// digits), two CTAs of 8 ranking warps per SM on smaller tiles, which the
// autotuner may pick where the arrays hold few tiles per SM; LB_SHAPE_4096,
// tiles that blocks of 4096 elements fit
template <typename F> static cudaError_t lb_dispatch_shape(int kb, int db, bool hasv, int shape, F &&f)
{
    using u64 = unsigned long long;
    if (shape == 2 && db == 8) {
        if (kb == 4)
            return hasv ? f.template operator()<uint32_t, true, 4096, 8>()
                        : f.template operator()<uint32_t, false, 8192, 8>();
        return hasv ? f.template operator()<u64, true, 4096, 8>() : f.template operator()<u64, false, 4096, 8>();
    }
    if (shape == LB_SHAPE_4096) {
        if (kb == 4)
            return hasv ? f.template operator()<uint32_t, true, 8192, 16>()
                        : f.template operator()<uint32_t, false, 16384, 16>();
        return hasv ? f.template operator()<u64, true, 4096, 16>() : f.template operator()<u64, false, 8192, 16>();
    }
    return lb_dispatch(kb, hasv, f);
}

} // namespace

bool lb_shape_differs(int db, int shape) { return shape == 2 && db == 8; }

uint32_t lb_tile(int kb, int db, bool hasv, int shape)
{
    uint32_t r = 0;
    lb_dispatch_shape(kb, db, hasv, shape,
                      [&]<typename KT, bool HASV, int TILE, int NW>() {
                          r = TILE;
                          return cudaSuccess;
                      });
    return r;
}

// ---------------------------------------------------------------- look-back ring
// Rows of the look-back ring: a power of two, no more than the tiles' power
// of two up to 512 rows, a quarter of it beyond (the tiles in flight at once,
// at most STAGES per SM, mostly fit; a tile whose slot is still in use waits
// for it), at most 2048 rows: a few MB whatever n.
static uint32_t ring_rows(size_t ntiles)
{
    constexpr uint32_t cap = 2048u;
    uint32_t r = 1;
    while (r < ntiles && r < 4 * cap)
        r <<= 1;
    if (r > 512)
        r = r / 4 > 512 ? r / 4 : 512u;
    return r < cap ? r : cap;
}

static size_t ring_bytes(size_t ntiles)
{
    const size_t r = ring_rows(ntiles);
    return r * 256 * 8 + r * 4;
}

template <typename KT> static void set_ring(LbArgs<KT> &a, void *mem, size_t ntiles, int pass)
{
    const uint32_t R = ring_rows(ntiles);
    a.ring = static_cast<unsigned long long *>(mem);
    a.done = reinterpret_cast<uint32_t *>(a.ring + size_t(R) * 256);
    a.rmask = R - 1;
    a.tagbase = uint32_t(pass + 1) << 24;
}

size_t grid_ring_bytes(const Geom &g)
{
    const uint32_t tile = lb_tile(g.kb, g.db, g.hasv, g.shape);
    return ring_bytes((g.n + tile - 1) / tile);
}

// ---------------------------------------------------------------- grid-layout Radsort
size_t grid_tab_words(const Geom &g) { return size_t(digit_passes(g.kb, g.db, false)) * GridTab::WORDS; }

const uint32_t *grid_skip_word(const Bufs &w, int pass)
{
    return w.tab + size_t(pass) * GridTab::WORDS + GridTab::HDR + TAB_SKIP;
}

cudaError_t launch_grid_tables(const Geom &g, const Bufs &w, uint32_t *pi, bool setup, cudaStream_t st)
{
    const uint32_t n = static_cast<uint32_t>(g.n), np = static_cast<uint32_t>(digit_passes(g.kb, g.db, g.whole));
    int blocks = setup ? static_cast<int>((g.npi + 1023) / 1024) : 0;
    if (blocks > 1024)
        blocks = 1024;
    auto go = [&]<typename KT>() {
        k_grid_tables<KT><<<np + blocks, 1024, 0, st>>>(w.hist, w.tab, 0u, np, n, g.lb, g.H, g.nA, g.npi,
                                                       static_cast<const KT *>(w.Ak), w.Av, static_cast<KT *>(w.Tk),
                                                       w.Tv, pi, w.P, w.state);
    };
    if (g.kb == 4)
        go.template operator()<uint32_t>();
    else
        go.template operator()<unsigned long long>();
    g_launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_grid_setup(const Geom &g, const Bufs &w, uint32_t *pi, cudaStream_t st)
{
    // cleared: the state, the tickets, the histograms (all digits' counts from
    // the input keys, before any block moves) and the look-back ring (no
    // tags), which lie in this order
    char *z0 = reinterpret_cast<char *>(w.state);
    cudaError_t e = cudaMemsetAsync(z0, 0, reinterpret_cast<char *>(w.status) + grid_ring_bytes(g) - z0, st);
    if (e != cudaSuccess)
        return e;
    e = launch_digit_hist(w.Ak, static_cast<uint32_t>(g.n), g.kb, by_bytes(g.db, g.whole), g.flt, w.hist, st);
    if (e != cudaSuccess)
        return e;
    return launch_grid_tables(g, w, pi, true, st);
}

cudaError_t launch_grid_prep(const Geom &g, const Bufs &w, const uint32_t *pi, uint32_t *pin, int pass,
                             cudaStream_t st)
{
    int blocks = static_cast<int>((g.npi + 255) / 256);
    if (blocks > num_sms() * 8)
        blocks = num_sms() * 8;
    k_grid_fill<<<blocks, 256, 0, st>>>(w.tab + size_t(pass) * GridTab::WORDS, static_cast<uint32_t>(g.n), g.lb, g.H,
                                        g.nA, g.npi, pi, pin);
    g_launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_grid_round(const Geom &g, const Bufs &w, const uint32_t *pi, uint32_t *pin, int pass,
                              cudaStream_t st)
{
    const uint32_t n = static_cast<uint32_t>(g.n);
    return lb_dispatch_shape(g.kb, g.db, g.hasv, g.shape,
                             [&]<typename KT, bool HASV, int TILE, int NW>() {
        using K = LbKernel<KT, HASV, TILE, NW, false>;
        const size_t ntiles = (g.n + TILE - 1) / TILE;
        const int grid = K::ctas(ntiles);
        if (grid < 0)
            return cudaErrorInvalidValue;
        LbArgs<KT> a{};
        a.Ak = static_cast<KT *>(w.Ak);
        a.Av = w.Av;
        a.Tk = static_cast<KT *>(w.Tk);
        a.Tv = w.Tv;
        a.pi = pi;
        a.pin = pin;
        a.tab = w.tab + size_t(pass) * GridTab::WORDS;
        a.hdr = a.tab + GridTab::HDR;
        set_ring(a, w.status, ntiles, pass);
        a.ticket = w.ctr + pass;
        a.n = n;
        a.ntiles = static_cast<uint32_t>(ntiles);
        a.H = g.H;
        a.nT = g.nT;
        a.npi = g.npi;
        a.lb = g.lb;
        if (g.flt)
            a.flt = (pass == 0 ? 1u : 0u) | (pass == digit_passes(g.kb, g.db, true) - 1 ? 2u : 0u);
        const DigitPass dp = digit_pass(g.kb, g.db, g.whole, pass);
        a.shift = dp.shift;
        a.mask = dp.mask();
        K::launch(grid, a, st);
        g_launches += 1;
        return cudaGetLastError();
    });
}

// ---------------------------------------------------------------- out-of-place comparator
// [counts | bucket starts | look-back ring | tickets]; the tables' sizes are
// those of sigma = 2^db
struct OopLayout {
    size_t off, ring, ctr, total;
};

static OopLayout oop_layout(size_t n, int kb, int db, bool hasv)
{
    const size_t sigma = size_t(1) << db, nt = (8 * kb + db - 1) / db;
    const uint32_t tile = lb_tile(kb, db, hasv, 0);
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t ring = ring_bytes((n + tile - 1) / tile);
    OopLayout L{};
    L.off = al(nt * sigma * 4);
    L.ring = L.off + al(nt * (sigma + 1) * 4);
    L.ctr = L.ring + al(ring > sigma * 8 ? ring : sigma * 8);
    L.total = L.ctr + al(64 * 4);
    return L;
}

size_t lsd_oop_scratch_bytes(size_t n, int kb, int db, bool hasv) { return oop_layout(n, kb, db, hasv).total; }

cudaError_t launch_lsd_oop_ws(void *keys, uint32_t *vals, void *keys_alt, uint32_t *vals_alt,
                              size_t n, int kb, int db, void *scratch, cudaStream_t st)
{
    if (n >= (size_t(1) << 31))
        return cudaErrorInvalidValue;
    const int np = kb; // whole sort: a pass per byte (an even number: the result ends in keys)
    const OopLayout L = oop_layout(n, kb, db, vals != nullptr);
    char *scr = static_cast<char *>(scratch);
    const bool own = scr == nullptr;
    cudaError_t e = cudaSuccess;
    if (own)
        e = cudaMallocAsync(reinterpret_cast<void **>(&scr), L.total, st);
    if (e != cudaSuccess)
        return e;
    uint32_t *hist = reinterpret_cast<uint32_t *>(scr), *off = reinterpret_cast<uint32_t *>(scr + L.off);
    uint32_t *ctr = reinterpret_cast<uint32_t *>(scr + L.ctr);
    // counts, ring and tickets cleared (the bucket starts between them too)
    e = cudaMemsetAsync(hist, 0, L.total, st);
    const uint32_t nn = static_cast<uint32_t>(n);
    if (e == cudaSuccess)
        e = launch_digit_hist(keys, nn, kb, true, false, hist, st);
    if (e == cudaSuccess) {
        k_offsets<<<np, 256, 0, st>>>(hist, off, nn);
        g_launches += 1;
        e = lb_dispatch(kb, vals != nullptr, [&]<typename KT, bool HASV, int TILE, int NW>() {
            using K = LbKernel<KT, HASV, TILE, NW, true>;
            const size_t ntiles = (n + TILE - 1) / TILE;
            const int grid = K::ctas(ntiles);
            if (grid < 0)
                return cudaErrorInvalidValue;
            KT *src = static_cast<KT *>(keys), *dst = static_cast<KT *>(keys_alt);
            uint32_t *vs = vals, *vd = vals_alt;
            for (int r = 0; r < np; ++r) {
                LbArgs<KT> a{};
                a.ik = src;
                a.iv = vs;
                a.ok = dst;
                a.ov = vd;
                a.tab = off + size_t(r) * 257;
                set_ring(a, scr + L.ring, ntiles, r);
                a.ticket = ctr + r;
                a.n = nn;
                a.ntiles = static_cast<uint32_t>(ntiles);
                const DigitPass dp = digit_pass(kb, db, true, r);
                a.shift = dp.shift;
                a.mask = dp.mask();
                K::launch(grid, a, st);
                g_launches += 1;
                std::swap(src, dst);
                std::swap(vs, vd);
            }
            return cudaGetLastError();
        });
    }
    cudaError_t e2 = own ? cudaFreeAsync(scr, st) : cudaSuccess;
    return e != cudaSuccess ? e : e2;
}

// ---------------------------------------------------------------- groups of arrays, 8-bit digits
// [alternate keys | alternate values | cleared: counts, tickets, look-back ring | bucket starts]
struct GroupLayout {
    size_t altv, hist, ctr, ring, tab, total;
    uint32_t ntiles;
};

static GroupLayout group_layout(const SegGroup &g, int kb, bool hasv)
{
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    GroupLayout L{};
    const uint32_t tile = lb_tile(kb, 8, hasv, 0);
    size_t el = 0;
    for (uint32_t i = 0; i < g.narr; ++i) {
        el += (size_t(g.len[i]) + 3) & ~size_t(3);
        L.ntiles += (g.len[i] + tile - 1) / tile;
    }
    size_t off = al(el * kb);
    L.altv = off;
    off += hasv ? al(el * 4) : 0;
    L.hist = off;
    off += al(size_t(g.narr) * kb * 256 * 4);
    L.ctr = off;
    off += al(64 * 4);
    L.ring = off;
    off += al(ring_bytes(L.ntiles));
    L.tab = off;
    off += al(size_t(g.narr) * kb * 257 * 4);
    L.total = off;
    return L;
}

size_t lsd_group_bytes(const SegGroup &g, int kb, bool hasv) { return group_layout(g, kb, hasv).total; }

cudaError_t launch_lsd_group(void *keys, uint32_t *vals, const SegGroup &g, int kb, void *pool, cudaStream_t st)
{
    const GroupLayout L = group_layout(g, kb, vals != nullptr);
    char *base = static_cast<char *>(pool);
    uint32_t *hist = reinterpret_cast<uint32_t *>(base + L.hist), *ctr = reinterpret_cast<uint32_t *>(base + L.ctr);
    uint32_t *tab = reinterpret_cast<uint32_t *>(base + L.tab);
    cudaError_t e = cudaMemsetAsync(hist, 0, L.tab - L.hist, st);
    if (e != cudaSuccess)
        return e;
    return lb_dispatch(kb, vals != nullptr, [&]<typename KT, bool HASV, int TILE, int NW>() {
        using C = Lb8Cfg<KT, HASV, TILE, NW, true>;
        const auto kern = k_lb_round8<KT, HASV, TILE, NW, true, true>;
        static DeviceOnce attr;
        const cudaError_t ea = attr.run([&] {
            cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
            if (r == cudaSuccess)
                r = cudaFuncSetAttribute(k_group_hist<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         4 * 256 * 32 * 4);
            return r;
        });
        if (ea != cudaSuccess)
            return ea;
        LbGroup in{}, out{}; // even rounds: from the arrays; odd rounds: back to them
        in.narr = g.narr;
        uint32_t tiles = 0, chunks = 0;
        size_t alt = 0;
        for (uint32_t i = 0; i < g.narr; ++i) {
            in.tile0[i] = tiles;
            in.len[i] = g.len[i];
            in.in[i] = g.off[i];
            in.out[i] = alt;
            tiles += (g.len[i] + TILE - 1) / TILE;
            chunks += (g.len[i] + GRP_CHUNK - 1) / GRP_CHUNK;
            alt += (size_t(g.len[i]) + 3) & ~size_t(3);
        }
        out = in;
        std::swap(out.in, out.out);
        constexpr int nt = int(sizeof(KT));
        k_group_hist<KT><<<dim3(chunks, nt / 4), 1024, 4 * 256 * 32 * 4, st>>>(static_cast<const KT *>(keys), in, hist);
        k_group_offsets<<<g.narr * nt, 256, 0, st>>>(hist, nt, g.narr, in, tab);
        const int sms = num_sms(), grid = tiles < uint32_t(sms) ? static_cast<int>(tiles) : sms;
        KT *alt_k = reinterpret_cast<KT *>(base);
        uint32_t *alt_v = HASV ? reinterpret_cast<uint32_t *>(base + L.altv) : nullptr;
        for (int r = 0; r < nt; ++r) {
            LbArgs<KT> a{};
            a.ik = r & 1 ? alt_k : static_cast<KT *>(keys);
            a.iv = r & 1 ? alt_v : vals;
            a.ok = r & 1 ? static_cast<KT *>(keys) : alt_k;
            a.ov = r & 1 ? vals : alt_v;
            a.tab = tab + size_t(r) * g.narr * 257;
            set_ring(a, base + L.ring, tiles, r);
            a.ticket = ctr + r;
            a.ntiles = tiles;
            a.shift = static_cast<uint32_t>(r * 8);
            a.mask = 255u;
            kern<<<grid, C::THREADS, C::SMEM, st>>>(a, r & 1 ? out : in);
        }
        g_launches += 2 + nt;
        return cudaGetLastError();
    });
}

cudaError_t launch_lsd_oop(void *keys, uint32_t *vals, void *keys_alt, uint32_t *vals_alt,
                           size_t n, int kb, int db, cudaStream_t st)
{
    return launch_lsd_oop_ws(keys, vals, keys_alt, vals_alt, n, kb, db, nullptr, st);
}

} // namespace rs
