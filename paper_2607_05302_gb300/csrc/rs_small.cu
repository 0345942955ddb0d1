// Short arrays in one launch (sm_103a): the whole array lives in the shared
// memory of one thread-block cluster of up to 16 CTAs, which runs every digit
// round of Alg. 1 there and writes the array back once.
//
// What bounds a short sort is launches and their latency: through the round
// kernel a sort of 1,000 keys is nine dependent launches and a stream-ordered
// allocation (59 us, 268 us when the allocation pool has given its memory
// back), one of 100,003 the same nine launches on 10 of 152 SMs (69 us).  Here
// it is one launch, with no memory but the array's own.  CTA r of the cluster
// holds positions [r P, (r + 1) P).  A round ranks the elements as the round
// kernel does (half-warps, one word per digit), exchanges the CTAs' digit
// counts through distributed shared memory, and scatters every element to its
// place in the cluster's other buffer, on whichever CTA that is.
// Measured (us; u32 + u32 with the copy of the input, workspace given, calls back
// to back; machines differ by a few percent): 1,000 24-26, 10,000 25, 24,576 29,
// 57,344 39, 106,496 53, 130,000 62-66, 155,648 68 (the round kernel takes 72-81
// from 155,649 to 200,003); u64 + u32 1,000 24-26, 24,576 57, 57,344 87, 57,345
// 116, 106,496 134-136.  Replayed as graphs, without the copy, where launches cost
// less: 12, 20, 24, 33, 48, 56-61, 63 (the round kernel 55-60) and 18, 52, 82,
// 110, 129.  Past 155,648, and 106,496 of 12 bytes, the array no longer fits the
// cluster; for the line with a workspace see small_sort_max.
#include "rs_common.cuh"
#include "rs_kernels.cuh"

namespace rs {

namespace {

constexpr int SM_T = 512;            // threads per CTA
constexpr int SM_ROWS = SM_T / 16;   // half-warps
constexpr int SM_MAXC = 16;          // CTAs of the largest cluster

// ITEMS elements per thread; odd, so that the two half-warps of a warp read
// different banks
template <typename KT, bool HASV, int ITEMS> struct SmCfg {
    static constexpr int P = ITEMS * SM_T;   // positions per CTA
    static constexpr int R = ITEMS * 16;     // elements per half-warp
    static_assert(ITEMS % 2 == 1, "odd");
    static constexpr bool PAIR = HASV && sizeof(KT) == 4; // keys and values as 8-byte words
    static constexpr size_t KB = size_t(P) * (PAIR ? 8 : sizeof(KT));
    static constexpr size_t BUF = KB + (HASV && !PAIR ? size_t(P) * 4 : 0);
    static constexpr size_t o_tab = 2 * BUF;                          // SM_ROWS x 256 words
    static constexpr size_t o_part = o_tab + size_t(SM_ROWS) * 256 * 4; // 2 x 256
    static constexpr size_t o_hist = o_part + 2 * 256 * 4;            // 256
    static constexpr size_t o_gst = o_hist + 256 * 4;                 // 256
    static constexpr size_t o_wsum = o_gst + 256 * 4;                 // 8 + 8
    static constexpr size_t SMEM = o_wsum + 64;
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
};

template <typename KT, bool HASV, int ITEMS, bool MULTI>
__global__ void __launch_bounds__(SM_T) k_small_sort(KT *keys, uint32_t *vals, uint32_t n, int flt)
{
    using C = SmCfg<KT, HASV, ITEMS>;
    constexpr uint32_t P = C::P;
    extern __shared__ __align__(16) unsigned char sm[];
    uint32_t *tab = reinterpret_cast<uint32_t *>(sm + C::o_tab);
    uint32_t *part = reinterpret_cast<uint32_t *>(sm + C::o_part);
    uint32_t *hist = reinterpret_cast<uint32_t *>(sm + C::o_hist);
    uint32_t *gst = reinterpret_cast<uint32_t *>(sm + C::o_gst);
    uint32_t *wsum = reinterpret_cast<uint32_t *>(sm + C::o_wsum);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, h = lane >> 4, l16 = lane & 15;
    const uint32_t rank = MULTI ? cluster_rank() : 0u, nc = MULTI ? cluster_size() : 1u;
    const uint32_t base = rank * P, cnt = n > base ? min(P, n - base) : 0u;
    const uint32_t sbase = smem_u32(sm);

    // ---- the array into the first buffer
    {
        KT *k0 = reinterpret_cast<KT *>(sm);
        uint2 *p0 = reinterpret_cast<uint2 *>(sm);
        uint32_t *v0 = reinterpret_cast<uint32_t *>(sm + C::KB);
        for (uint32_t i = tid; i < cnt; i += SM_T) {
            KT k = keys[base + i];
            if constexpr (sizeof(KT) == 4)
                if (flt)
                    k = float_to_ordered(k);
            if constexpr (C::PAIR) {
                p0[i] = make_uint2(k, vals[base + i]);
            } else {
                k0[i] = k;
                if (HASV)
                    v0[i] = vals[base + i];
            }
        }
    }
    for (int i = tid; i < SM_ROWS * 256; i += SM_T)
        tab[i] = 0u;
    __syncthreads();

    uint32_t *row = tab + (2 * warp + h) * 256;
    const uint32_t eh = uint32_t((2 * warp + h) * C::R + l16);
    const int c = tid & 255, p = tid >> 8; // the column passes' bucket and half of the rows
    uint32_t cur = 0;                      // the buffer that holds the sequence
    for (uint32_t shift = 0; shift < 8 * sizeof(KT); shift += 8) {
        const unsigned char *src = sm + cur * C::BUF;
        const uint32_t dst = sbase + (cur ^ 1u) * uint32_t(C::BUF);
        // ---- 1. elements into registers, stable ranks within the half-warp
        KT key[ITEMS];
        uint32_t val[HASV ? ITEMS : 1], rk[(ITEMS + 1) / 2];
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t e = eh + it * 16;
            if constexpr (C::PAIR) {
                const uint2 x = reinterpret_cast<const uint2 *>(src)[e];
                key[it] = x.x;
                val[it] = x.y;
            } else {
                key[it] = reinterpret_cast<const KT *>(src)[e];
                if (HASV)
                    val[it] = reinterpret_cast<const uint32_t *>(src + C::KB)[e];
            }
        }
        rank_half_warp<ITEMS>(row, [&](int it) { return digit_of(key[it], shift, 255u); },
                              [&](int it) { return eh + it * 16 < cnt; }, rk);
        __syncthreads();
        // ---- 2. the CTA's counts per digit, and their exchange
        uint32_t *col = tab + p * (SM_ROWS / 2) * 256 + c;
        uint32_t hc[SM_ROWS / 4], sum = 0;
#pragma unroll
        for (int r = 0; r < SM_ROWS / 2; r += 2) {
            const uint32_t x = col[r * 256] >> 16, y = col[(r + 1) * 256] & 0xFFFF0000u;
            hc[r >> 1] = x | y;
            sum += x + (y >> 16);
        }
        part[p * 256 + c] = sum;
        __syncthreads();
        uint32_t tot = 0, below = 0;
        if (p == 0) {
            tot = sum + part[256 + c];
            if (MULTI)
                hist[c] = tot;
        }
        if constexpr (MULTI) {
            cluster_sync();
            if (p == 0) {
                const uint32_t ha = sbase + uint32_t(C::o_hist) + c * 4;
                uint32_t all = 0;
#pragma unroll 8
                for (uint32_t q = 0; q < nc; ++q) {
                    const uint32_t x = ld_cluster(cluster_addr(ha, q));
                    all += x;
                    below += q < rank ? x : 0u;
                }
                tot = all;
            }
        }
        // ---- 3. each digit's start over the whole array, then each
        // half-warp's
        if (p == 0) {
            const uint32_t inc = warp_incl_scan(tot);
            if (lane == 31)
                wsum[warp] = inc;
            gst[c] = inc - tot + below;
        }
        // (one digit for the whole array: the round is the identity)
        const bool skip = __syncthreads_or(p == 0 && tot == n);
        if (skip) {
            // this warp's words for the next round
            __syncthreads();
            uint4 *z = reinterpret_cast<uint4 *>(tab + 2 * warp * 256);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                z[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
            if constexpr (MULTI)
                cluster_sync();
            else
                __syncthreads();
            continue;
        }
        uint32_t run = gst[c] + (p ? part[c] : 0u);
#pragma unroll
        for (int w = 0; w < 7; ++w)
            run += w < (c >> 5) ? wsum[w] : 0u;
#pragma unroll
        for (int r = 0; r < SM_ROWS / 2; ++r) {
            col[r * 256] = run;
            run += (r & 1) ? hc[r >> 1] >> 16 : hc[r >> 1] & 0xFFFFu;
        }
        __syncthreads();
        // ---- 4. every element to its place in the cluster's other buffer
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            const uint32_t e = eh + it * 16;
            if (e >= cnt)
                continue;
            const uint32_t pos =
                row[digit_of(key[it], shift, 255u)] + ((it & 1) ? rk[it >> 1] >> 16 : rk[it >> 1] & 0xFFFFu);
            if (pos >= n) { // only a broken scan gets here
                set_status(ST_INTERNAL);
                continue;
            }
            if constexpr (MULTI) {
                const uint32_t q = pos / P, l = pos - q * P;
                if constexpr (C::PAIR) {
                    st_cluster(cluster_addr(dst + l * 8, q), make_uint2(key[it], val[it]));
                } else {
                    st_cluster(cluster_addr(dst + l * uint32_t(sizeof(KT)), q), key[it]);
                    if (HASV)
                        st_cluster(cluster_addr(dst + uint32_t(C::KB) + l * 4, q), val[it]);
                }
            } else {
                unsigned char *d = sm + (cur ^ 1u) * C::BUF;
                if constexpr (C::PAIR) {
                    reinterpret_cast<uint2 *>(d)[pos] = make_uint2(key[it], val[it]);
                } else {
                    reinterpret_cast<KT *>(d)[pos] = key[it];
                    if (HASV)
                        reinterpret_cast<uint32_t *>(d + C::KB)[pos] = val[it];
                }
            }
        }
        __syncwarp();
        // this warp's words for the next round
        uint4 *z = reinterpret_cast<uint4 *>(tab + 2 * warp * 256);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            z[i * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
        if constexpr (MULTI)
            cluster_sync();
        else
            __syncthreads();
        cur ^= 1u;
    }

    // ---- the sorted array back
    const unsigned char *src = sm + cur * C::BUF;
    for (uint32_t i = tid; i < cnt; i += SM_T) {
        KT k;
        if constexpr (C::PAIR) {
            const uint2 x = reinterpret_cast<const uint2 *>(src)[i];
            k = x.x;
            vals[base + i] = x.y;
        } else {
            k = reinterpret_cast<const KT *>(src)[i];
            if (HASV)
                vals[base + i] = reinterpret_cast<const uint32_t *>(src + C::KB)[i];
        }
        if constexpr (sizeof(KT) == 4)
            if (flt)
                k = ordered_to_float(k);
        keys[base + i] = k;
    }
}

// Launches with the smallest cluster that holds n; cudaErrorNotSupported where
// the device has no room for the largest one.
template <typename KT, bool HASV, int ITEMS, bool MULTI>
cudaError_t small_launch(void *keys, uint32_t *vals, uint32_t n, int flt, cudaStream_t st)
{
    using C = SmCfg<KT, HASV, ITEMS>;
    const auto kern = k_small_sort<KT, HASV, ITEMS, MULTI>;
    const auto config = [st](uint32_t ctas, cudaLaunchAttribute *at) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(SM_T);
        cfg.dynamicSmemBytes = C::SMEM;
        cfg.stream = st;
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = ctas;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = MULTI ? 1 : 0;
        return cfg;
    };
    static DeviceOnce attr;
    const cudaError_t ea = attr.run([&] {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
        if (e == cudaSuccess && MULTI)
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess && MULTI) {
            cudaLaunchAttribute at{};
            const cudaLaunchConfig_t cfg = config(SM_MAXC, &at);
            int clusters = 0;
            e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
            if (e == cudaSuccess && clusters < 1)
                e = cudaErrorNotSupported;
        }
        return e;
    });
    if (ea != cudaSuccess)
        return ea;
    uint32_t ctas = 1;
    while (size_t(ctas) * C::P < n)
        ctas <<= 1;
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = config(ctas, &at);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<KT *>(keys), vals, n, flt);
    if (e == cudaSuccess)
        g_launches += 1;
    return e;
}

// the most elements per thread that two buffers leave room for
constexpr int small_items(int kb, bool hasv) { return kb + (hasv ? 4 : 0) <= 8 ? 19 : 13; }

template <typename KT, bool HASV>
cudaError_t small_dispatch(void *keys, uint32_t *vals, uint32_t n, int flt, cudaStream_t st)
{
    constexpr int BIG = small_items(int(sizeof(KT)), HASV);
    // few elements per thread rank faster, few CTAs exchange less: one CTA
    // up to 7 elements a thread, then as few elements as 16 CTAs allow
    if (n <= 3 * SM_T)
        return small_launch<KT, HASV, 3, false>(keys, vals, n, flt, st);
    if (n <= 7 * SM_T)
        return small_launch<KT, HASV, 7, false>(keys, vals, n, flt, st);
    if (n <= SM_MAXC * 3 * SM_T)
        return small_launch<KT, HASV, 3, true>(keys, vals, n, flt, st);
    if (n <= SM_MAXC * 7 * SM_T)
        return small_launch<KT, HASV, 7, true>(keys, vals, n, flt, st);
    if (BIG > 13 && n <= SM_MAXC * 13 * SM_T)
        return small_launch<KT, HASV, 13, true>(keys, vals, n, flt, st);
    return small_launch<KT, HASV, BIG, true>(keys, vals, n, flt, st);
}

} // namespace

unsigned take_status_small() { return take_status_word(); }

// The longest array sorted here.  12-byte elements scatter two words each across
// the cluster, and past 7 a thread the round kernel is faster where it has its
// workspace: 57,345 to 106,496 u64 + u32 111-118 us a call back to back against
// 116-136 here, as graphs 82-88 against 110-130.  A call that has to allocate
// the workspace still goes here: alone, after the pool has given its memory
// back, 119-139 against 220-230.
uint32_t small_sort_max(int kb, bool hasv, bool workspace)
{
    const int items = small_items(kb, hasv);
    return uint32_t(SM_MAXC * SM_T * (items == 13 && workspace ? 7 : items));
}

cudaError_t launch_small_sort(void *keys, uint32_t *vals, uint32_t n, int kb, bool flt, cudaStream_t st)
{
    using u64 = unsigned long long;
    if (kb == 4)
        return vals ? small_dispatch<uint32_t, true>(keys, vals, n, flt, st)
                    : small_dispatch<uint32_t, false>(keys, vals, n, flt, st);
    return vals ? small_dispatch<u64, true>(keys, vals, n, 0, st) : small_dispatch<u64, false>(keys, vals, n, 0, st);
}

} // namespace rs
