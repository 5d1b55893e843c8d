// util.cu -- kernel time-order check and permutation.
#include <algorithm>

#include "sort.cuh"
#include "util.cuh"

namespace opattr {

constexpr int CHK_THREADS = 256;

// Tiles of CHK_TILE consecutive kernels, a block at a time, each thread taking
// two groups of eight consecutive kernels per tile (16-byte loads when the
// arrays allow) and comparing each (start, stream) with its successor; min /
// max and the order flag are reduced per block and published with one atomic
// each.
constexpr int CHK_G = 8;
constexpr int CHK_TILE = 2 * CHK_THREADS * CHK_G;
__global__ void __launch_bounds__(CHK_THREADS) k_check_kernel_order(const uint8_t *__restrict__ stream,
                                                                    const int64_t *__restrict__ start, int64_t n,
                                                                    int vec, DevStatus *st) {
    pdl_wait();
    __shared__ long long smin[CHK_THREADS / 32], smax[CHK_THREADS / 32];
    __shared__ int sbad[CHK_THREADS / 32];
    long long mn = LLONG_MAX, mx = LLONG_MIN;
    int unsorted = 0;
    const int64_t ntiles = (n + CHK_TILE - 1) / CHK_TILE;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        for (int r = 0; r < 2; ++r) {
            const int64_t i0 = (tile * (CHK_TILE / CHK_G) + r * CHK_THREADS + threadIdx.x) * CHK_G;
            if (i0 >= n) continue;
            long long t[CHK_G + 1];
            unsigned s[CHK_G + 1];
            if (vec && i0 + CHK_G <= n) {
                const longlong2 *p = reinterpret_cast<const longlong2 *>(start + i0);
#pragma unroll
                for (int q = 0; q < CHK_G / 2; ++q) {
                    const longlong2 x = p[q];
                    t[2 * q] = x.x;
                    t[2 * q + 1] = x.y;
                }
                const uint2 w = *reinterpret_cast<const uint2 *>(stream + i0);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    s[u] = (w.x >> (8 * u)) & 0xFFu;
                    s[4 + u] = (w.y >> (8 * u)) & 0xFFu;
                }
            } else {
#pragma unroll
                for (int u = 0; u < CHK_G; ++u) {
                    t[u] = i0 + u < n ? start[i0 + u] : LLONG_MAX;
                    s[u] = i0 + u < n ? stream[i0 + u] : 255u;
                }
            }
            t[CHK_G] = i0 + CHK_G < n ? start[i0 + CHK_G] : LLONG_MAX;
            s[CHK_G] = i0 + CHK_G < n ? stream[i0 + CHK_G] : 255u;
#pragma unroll
            for (int u = 0; u < CHK_G; ++u) {
                if (i0 + u >= n) break;
                mn = t[u] < mn ? t[u] : mn;
                mx = t[u] > mx ? t[u] : mx;
                if (i0 + u + 1 < n) unsorted |= (t[u + 1] < t[u]) || (t[u + 1] == t[u] && s[u + 1] < s[u]);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        long long a = __shfl_xor_sync(0xffffffffu, mn, o), b = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = a < mn ? a : mn;
        mx = b > mx ? b : mx;
    }
    unsorted = __any_sync(0xffffffffu, unsorted);
    if (lane_id() == 0) {
        smin[threadIdx.x >> 5] = mn;
        smax[threadIdx.x >> 5] = mx;
        sbad[threadIdx.x >> 5] = unsorted;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int bad = 0;
        for (int w = 0; w < CHK_THREADS / 32; ++w) {
            mn = smin[w] < mn ? smin[w] : mn;
            mx = smax[w] > mx ? smax[w] : mx;
            bad |= sbad[w];
        }
        atomicMin(&st->mm[MM_KSTART_MIN], mn);
        atomicMax(&st->mm[MM_KSTART_MAX], mx);
        if (bad) set_flag(st, F_K_UNSORTED);
    }
}

void check_kernel_order(Ctx &c, const uint8_t *stream, const int64_t *start, int64_t n) {
    if (n <= 0) return;
    const int vec = ((reinterpret_cast<uintptr_t>(start) & 15) == 0) && ((reinterpret_cast<uintptr_t>(stream) & 7) == 0);
    launch(c, "check_kernel_order", k_check_kernel_order, dim3(grid_for(n, CHK_TILE, REDUCE_GRID)),
           dim3(CHK_THREADS), 0, stream, start, n, vec, c.d_status);
}

// ------------------------------------------------------------------ time sort
// Records sorted by a time key, ties by index: the key's high bits split the
// records over buckets of up to BK_TARGET on average (a count, a scan of the
// counts, a scatter in any order), then a block sorts each bucket in shared
// memory by spreading it over BK_BINS bins of the bucket's span and sorting
// every bin, a few records each, by key and index.  Two reads and two writes of
// 8 bytes per record, where the radix sort makes a pass of 24 bytes per eight
// key bits.  Times crowd when a trace has long gaps or many equal times: a
// bucket above BK_CAP records or a bin above BK_BIN_MAX sets *crowded, and the
// radix sort does the whole again.
//
// 6M kernel records in no order: 16 us to count, 77 to scatter (bound by the
// scattered 8-byte writes), 90 to sort the buckets (shared-memory latency),
// against 115 us for each of five radix passes.
//
// An entry holds 32 bits of key, so the span of the keys sets how many buckets
// there are at least, however few the records: 2^(bits - 32) of them.  A bucket
// costs its block some 12 ns whatever it holds.  Up to BK_FEW buckets, or one to
// BK_LEAST records, that is less than radix passes: 300,000 records whose keys span
// 2^44 / 2^46 / 2^47 values 153 / 300 / 495 us by buckets and 206 by radix, 4M 298 /
// 464 / 692 and 470; 3,000 with 4,096 buckets 126 and 170.
constexpr int BK_THREADS = 512, BK_ITEMS = 16, BK_CAP = BK_THREADS * BK_ITEMS, BK_BIN_BITS = 12,
              BK_BINS = 1 << BK_BIN_BITS;
constexpr int BK_TARGET = 3072;
constexpr int BK_BIN_MAX = 64;
constexpr int64_t BK_FEW = 4096, BK_LEAST = 256;
constexpr int64_t BK_MAX = 32 * 1024;        // buckets: their counts fit a block's shared memory and one block's scan

// Each block counts an equal share of the records in shared memory (global
// counters take few, coalesced additions: single ones ran at 50 a nanosecond).
template <typename Key>
__global__ void __launch_bounds__(BK_THREADS) k_bucket_count(Key key, int64_t n, int shift, int nb,
                                                             uint32_t *__restrict__ cnt) {
    pdl_wait();
    extern __shared__ uint32_t bk[];
    for (int i = threadIdx.x; i < nb; i += BK_THREADS) bk[i] = 0;
    __syncthreads();
    const int64_t share = (n + gridDim.x - 1) / gridDim.x, i0 = share * blockIdx.x;
    const int64_t i1 = i0 + share < n ? i0 + share : n;
#pragma unroll 4
    for (int64_t i = i0 + threadIdx.x; i < i1; i += BK_THREADS) atomicAdd(&bk[key(i) >> shift], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += BK_THREADS)
        if (bk[i]) atomicAdd(&cnt[i], bk[i]);
}
// Bucket b fills [off[b], off[b + 1]): entries (key below `shift`) << 32 | i;
// leaves off[b] at the bucket's end.  Same shares: counted again, room taken in
// every bucket at once, then handed out.
template <typename Key>
__global__ void __launch_bounds__(BK_THREADS) k_bucket_scatter(Key key, int64_t n, int shift, int nb,
                                                               uint32_t *__restrict__ off,
                                                               uint64_t *__restrict__ out) {
    pdl_wait();
    extern __shared__ uint32_t bk[];
    for (int i = threadIdx.x; i < nb; i += BK_THREADS) bk[i] = 0;
    __syncthreads();
    const int64_t share = (n + gridDim.x - 1) / gridDim.x, i0 = share * blockIdx.x;
    const int64_t i1 = i0 + share < n ? i0 + share : n;
#pragma unroll 4
    for (int64_t i = i0 + threadIdx.x; i < i1; i += BK_THREADS) atomicAdd(&bk[key(i) >> shift], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += BK_THREADS)
        if (bk[i]) bk[i] = atomicAdd(&off[i], bk[i]);
    __syncthreads();
    const uint64_t low = (1ull << shift) - 1;
#pragma unroll 4
    for (int64_t i = i0 + threadIdx.x; i < i1; i += BK_THREADS) {
        const uint64_t k = key(i);
        out[atomicAdd(&bk[k >> shift], 1u)] = (k & low) << 32 | (uint32_t)i;
    }
}
__global__ void __launch_bounds__(BK_THREADS) k_bucket_sort(const uint64_t *__restrict__ in,
                                                            const uint32_t *__restrict__ end, int shift,
                                                            uint64_t *__restrict__ keys, uint32_t *__restrict__ perm,
                                                            uint32_t *crowded) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char bk_smem[];
    uint64_t *buf = reinterpret_cast<uint64_t *>(bk_smem);              // [BK_CAP]
    uint32_t *bin = reinterpret_cast<uint32_t *>(buf + BK_CAP);         // [BK_BINS]
    __shared__ uint32_t wbuf[33];
    const int64_t b = blockIdx.x;
    const uint32_t s0 = b ? end[b - 1] : 0u, m = end[b] - s0;
    if (m == 0) return;
    if (m > (uint32_t)BK_CAP) {
        if (threadIdx.x == 0) *crowded = 1u;
        return;
    }
    constexpr int PER = BK_BINS / BK_THREADS;
    for (int i = threadIdx.x; i < BK_BINS; i += BK_THREADS) bin[i] = 0;
    __syncthreads();
    // bins by the bits below the bucket's: the top BK_BIN_BITS of them
    const int down = 32 + (shift > BK_BIN_BITS ? shift - BK_BIN_BITS : 0);
    uint64_t v[BK_ITEMS];
    uint32_t r[BK_ITEMS];
#pragma unroll
    for (int i = 0; i < BK_ITEMS; ++i) {
        const uint32_t j = i * BK_THREADS + threadIdx.x;
        if (j >= m) continue;
        v[i] = in[s0 + j];
        r[i] = atomicAdd(&bin[v[i] >> down], 1u);
    }
    __syncthreads();
    uint32_t c[PER], sum = 0;
    bool full = false;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        c[q] = bin[threadIdx.x * PER + q];
        full |= c[q] > (uint32_t)BK_BIN_MAX;
        sum += c[q];
    }
    uint32_t ex = block_exclusive_scan<uint32_t>(sum, wbuf, (uint32_t *)nullptr);
    const uint32_t first = ex;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        bin[threadIdx.x * PER + q] = ex;
        ex += c[q];
    }
    if (__syncthreads_or(full)) {
        if (threadIdx.x == 0) *crowded = 1u;
        return;
    }
#pragma unroll
    for (int i = 0; i < BK_ITEMS; ++i)
        if (i * BK_THREADS + threadIdx.x < m) buf[bin[v[i] >> down] + r[i]] = v[i];
    __syncthreads();
    // each thread's bins, one after another: insertion sort (unique entries)
    for (uint32_t q = 0, a = first; q < (uint32_t)PER; ++q) {
        const uint32_t z = q + 1 < (uint32_t)PER ? bin[threadIdx.x * PER + q + 1] : ex;
        for (uint32_t i = a + 1; i < z; ++i) {
            const uint64_t x = buf[i];
            uint32_t j = i;
            for (; j > a && buf[j - 1] > x; --j) buf[j] = buf[j - 1];
            buf[j] = x;
        }
        a = z;
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < m; j += BK_THREADS) {
        const uint64_t x = buf[j];
        keys[s0 + j] = (uint64_t)b << shift | x >> 32;
        perm[s0 + j] = (uint32_t)x;
    }
}
template <typename Key>
__global__ void k_write_keys(Key key, int64_t n, uint64_t *__restrict__ keys) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = key(i);
}
// The two halves of a key that does not fit 64 bits: what follows the time, and
// then the times in the order that this gave.
template <typename Key>
__global__ void k_write_low(Key key, int64_t n, uint64_t *__restrict__ keys) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = key.low(i);
}
template <typename Key>
__global__ void k_gather_times(Key key, const uint32_t *__restrict__ perm, int64_t n, uint64_t *__restrict__ keys) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = key.time(perm[i]);
}

size_t time_sort_scratch(int64_t n) {
    Need nd;
    nd.add<uint64_t>(n).add<uint64_t>(n).add<uint32_t>(n).add<uint32_t>(n);
    nd.add<uint32_t>(std::max<int64_t>(radix_hist_elems(n), BK_MAX + 1));
    nd.add<uint32_t>(scan_scratch_elems(std::max<int64_t>(radix_hist_elems(n), BK_MAX + 1)));
    return nd.bytes;
}

// Records 0 .. n - 1 by key(i) = time(i) << bits | low(i), with time(i) at most
// `span`; *keys receives the sorted keys.  Where span << bits does not fit 64
// bits the sort goes by low(i) first and by time(i) then, and *keys is NULL.
template <typename Key>
static opattr_status time_sort(Ctx &c, Arena &a, Key key, int64_t n, uint64_t span, uint64_t **keys, uint32_t **perm) {
    const int64_t hist_n = std::max<int64_t>(radix_hist_elems(n), BK_MAX + 1);
    uint64_t *k0 = a.take<uint64_t>(n), *k1 = a.take<uint64_t>(n);
    uint32_t *v0 = a.take<uint32_t>(n), *v1 = a.take<uint32_t>(n);
    uint32_t *hist = a.take<uint32_t>(hist_n), *part = a.take<uint32_t>(scan_scratch_elems(hist_n));
    if (!k0 || !k1 || !v0 || !v1 || !hist || !part) return OPATTR_E_OOM;
    if (bits_for(span) + key.bits > 64) {
        const dim3 g(grid_for(n, 256, 65535));
        uint64_t *k = nullptr;
        uint32_t *v = nullptr;
        launch(c, "time_keys", k_write_low<Key>, g, dim3(256), 0, key, n, k0);
        radix_sort_pairs<uint64_t>(c, k0, v0, k1, v1, n, key.bits, true, hist, part, &k, &v);
        launch(c, "time_keys", k_gather_times<Key>, g, dim3(256), 0, key, (const uint32_t *)v, n, k);
        radix_sort_pairs<uint64_t>(c, k, v, k == k0 ? k1 : k0, v == v0 ? v1 : v0, n, bits_for(span), false, hist, part,
                                   &k, perm);
        *keys = nullptr;
        return OPATTR_OK;
    }
    // no key is above it: the bucket counts in shared memory are indexed by the key's high bits
    const uint64_t top = span << key.bits | ((1ull << key.bits) - 1);
    // widest buckets of BK_TARGET records on average whose span fits the entries' 32 bits
    int shift = 32;
    while (shift > 0 && (int64_t)(top >> shift) + 1 < (n + BK_TARGET - 1) / BK_TARGET) --shift;
    const int64_t nb = (int64_t)(top >> shift) + 1;
    if (c.host_mapped && nb <= std::min(BK_MAX, std::max(BK_FEW, n / BK_LEAST))) {
        const int sms = sm_count(c);
        const size_t smem = sizeof(uint32_t) * nb, sort_smem = sizeof(uint64_t) * BK_CAP + sizeof(uint32_t) * BK_BINS;
        const dim3 g(grid_for(n, BK_THREADS * 8, (smem > 64 * 1024 ? 1 : 3) * sms));
        cudaFuncSetAttribute(k_bucket_count<Key>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(4 * BK_MAX));
        cudaFuncSetAttribute(k_bucket_scatter<Key>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(4 * BK_MAX));
        cudaFuncSetAttribute(k_bucket_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sort_smem);
        uint32_t *crowded = hist + nb;                // after the counts: hist holds BK_MAX + 1 at least
        const ZeroRun z{hist, nb + 1};
        opattr_status st = zero_runs(c, 1, &z);
        if (st) return st;
        launch(c, "bucket_count", k_bucket_count<Key>, g, dim3(BK_THREADS), smem, key, n, shift, (int)nb, hist);
        scan_exclusive_u32(c, hist, hist, nb, part, nullptr);
        launch(c, "bucket_scatter", k_bucket_scatter<Key>, g, dim3(BK_THREADS), smem, key, n, shift, (int)nb, hist, k0);
        launch(c, "bucket_sort", k_bucket_sort, dim3((unsigned)nb), dim3(BK_THREADS), sort_smem, (const uint64_t *)k0,
               (const uint32_t *)hist, shift, k1, v1, crowded);
        const SmallCopy verdict{c.h_small, crowded, sizeof(uint32_t)};
        if ((st = read_status(c, 1, &verdict))) return st;
        *keys = k1;
        *perm = v1;
        if (!c.h_small[0]) return OPATTR_OK;
    }
    launch(c, "time_keys", k_write_keys<Key>, dim3(grid_for(n, 256, 65535)), dim3(256), 0, key, n, k0);
    radix_sort_pairs<uint64_t>(c, k0, v0, k1, v1, n, bits_for(top), true, hist, part, keys, perm);
    return OPATTR_OK;
}

struct KernelTimeKey {
    const int64_t *start;
    const uint8_t *stream, *scmap;      // scmap may be NULL
    long long tmin;
    int bits;
    __device__ __forceinline__ uint64_t time(int64_t i) const { return (uint64_t)start[i] - (uint64_t)tmin; }
    __device__ __forceinline__ unsigned low(int64_t i) const {
        const unsigned s = stream[i];
        return scmap ? scmap[s] : s;
    }
    __device__ __forceinline__ uint64_t operator()(int64_t i) const { return time(i) << bits | low(i); }
};
opattr_status kernel_time_order(Ctx &c, Arena &a, const uint8_t *stream, const int64_t *start, int64_t n,
                                uint32_t **order, const uint8_t *scmap, int stream_bits, uint64_t **keys) {
    const long long tmin = c.h_status->mm[MM_KSTART_MIN], tmax = c.h_status->mm[MM_KSTART_MAX];
    uint64_t *k = nullptr;
    const opattr_status st = time_sort(c, a, KernelTimeKey{start, stream, scmap, tmin, scmap ? stream_bits : 8}, n,
                                       (uint64_t)tmax - (uint64_t)tmin, &k, order);
    if (st) return st;
    if (keys && !k) return OPATTR_E_INVALID_ARG;
    if (keys) *keys = k;
    return OPATTR_OK;
}

// The order key of range i: its start, then its depth, so that parents come
// before children that start with them, then 0 for a zero-length range and 1
// for a longer one.  Within a level of laminar ranges two ranges share a start
// only if all but the last of them have zero length, so a stable sort on this
// key puts every level in (start, end, index) order -- the order of Algorithm
// 2's one representative per depth; two longer ranges sharing a start in one
// level are out of that order only when they overlap, which the laminar
// checks report.
struct RangeTimeKey {
    static constexpr int bits = RANGE_KEY_SHIFT;
    const int64_t *start, *end;
    const uint8_t *depth;
    long long tmin;
    __device__ __forceinline__ uint64_t time(int64_t i) const { return (uint64_t)start[i] - (uint64_t)tmin; }
    __device__ __forceinline__ unsigned low(int64_t i) const { return depth[i] << 1 | (end[i] > start[i] ? 1u : 0u); }
    __device__ __forceinline__ uint64_t operator()(int64_t i) const { return time(i) << bits | low(i); }
};
opattr_status range_time_order(Ctx &c, Arena &a, const int64_t *start, const int64_t *end, const uint8_t *depth,
                               int64_t n, long long tmin, long long tmax, uint32_t **order, uint64_t **keys) {
    return time_sort(c, a, RangeTimeKey{start, end, depth, tmin}, n, (uint64_t)tmax - (uint64_t)tmin, keys, order);
}

}  // namespace opattr
