// match.cu -- Algorithm 1 (invocation-order matching, Sec. 3.3) and layer
// deduplication broadcast (Sec. 3.7) on the GPU.
//
// Fast path.  When the replayed kernels, in time order, carry exactly the
// names of the ncu rows in array order, launch i pairs with row i and no
// ordinal is computed: one pass compares the two name arrays and writes the
// identity.  Exports in time order with ncu replaying the same launches hit
// this path.  With per-stream rows (the rows of each stream in launch order,
// streams one after another) the same test runs on the replayed kernels and
// the rows each partitioned stably by stream.
//
// General path.  Ordinals come from one stable radix sort by name of the
// replayed kernels in time order followed by the ncu rows in array order: a
// name's run of kernels, in launch order, is followed by its run of rows, in
// launch order, and the join is row = rows_of_name[position in the run], subject
// to the mismatch mode.  Dedup positions come from a stable partition of the
// layer-tagged kernels by layer id.
#include <algorithm>

#include "sort.cuh"
#include "util.cuh"

namespace opattr {

// ------------------------------------------------------------------ fast path
// Whether the identity pass may use 16-byte accesses (every array aligned).
static int identity_vec(const void *kname, const void *nname, const void *out_idx, const void *out_kind) {
    auto al = [](const void *p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
    return al(kname, 16) && al(nname, 16) && al(out_idx, 16) && al(out_kind, 4);
}
__global__ void k_match_identity(const uint32_t *__restrict__ kname, const uint32_t *__restrict__ nname, int64_t n,
                                 int32_t *__restrict__ out_idx, uint8_t *__restrict__ out_kind, int vec,
                                 DevStatus *st) {
    pdl_wait();
    constexpr int U = 4;                    // elements per thread per round, loads issued together
    int bad = 0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * U;
    for (int64_t base = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * U; base < n; base += stride) {
        if (vec && base + U <= n) {         // 16-byte loads and stores
            const uint4 a = *reinterpret_cast<const uint4 *>(kname + base);
            const uint4 b = *reinterpret_cast<const uint4 *>(nname + base);
            bad |= (a.x != b.x) | (a.y != b.y) | (a.z != b.z) | (a.w != b.w);
            const int32_t i0 = (int32_t)base;
            *reinterpret_cast<int4 *>(out_idx + base) = make_int4(i0, i0 + 1, i0 + 2, i0 + 3);
            if (out_kind) *reinterpret_cast<uint32_t *>(out_kind + base) = 0x01010101u;
            continue;
        }
        uint32_t a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            a[u] = base + u < n ? kname[base + u] : 0u;
            b[u] = base + u < n ? nname[base + u] : 0u;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (base + u >= n) continue;
            bad |= a[u] != b[u];
            out_idx[base + u] = (int32_t)(base + u);
            if (out_kind) out_kind[base + u] = 1;
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_flag(st, F_NAMES_DIFFER);
}

// replayed kernels in time order (list rk) against rows 0..n-1
__global__ void k_match_identity_list(const uint32_t *__restrict__ rk, const uint32_t *__restrict__ kname,
                                      const uint32_t *__restrict__ nname, int64_t n, int32_t *__restrict__ out_idx,
                                      uint8_t *__restrict__ out_kind, DevStatus *st) {
    pdl_wait();
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t k = rk[i];
        bad |= kname[k] != nname[i];
        out_idx[k] = (int32_t)i;
        if (out_kind) out_kind[k] = 1;
    }
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_flag(st, F_NAMES_DIFFER);
}

// Per-stream rows.  Replayed kernel j (kernel rk[j], or j when rk is null)
// takes position dest of the replayed kernels partitioned stably by stream;
// the row at that position of the rows partitioned the same way is pn[dest].
// The pairing holds when name and stream agree everywhere; name ids must
// also fit in 24 bits, as (name, stream) keys require.
struct StreamDigit {
    const uint32_t *rk;
    const uint8_t *stream;
    __device__ __forceinline__ unsigned operator()(int64_t j) const { return stream[rk ? rk[j] : (uint32_t)j]; }
};
struct StreamPairs {
    const uint32_t *rk, *pn, *kname, *nname;
    const uint8_t *kstream, *nstream;
    int32_t *out_idx;
    uint8_t *out_kind;
    DevStatus *st;
    __device__ __forceinline__ unsigned operator()(int64_t j, uint32_t dest, unsigned) const {
        const uint32_t k = rk ? rk[j] : (uint32_t)j;
        const uint32_t r = pn[dest];
        const uint32_t x = kname[k], y = nname[r];
        out_idx[k] = (int32_t)r;
        if (out_kind) out_kind[k] = 1;
        return (x != y || kstream[k] != nstream[r] ? 1u : 0u) | ((x | y) >> 24 != 0 ? 2u : 0u);
    }
    __device__ __forceinline__ void done(unsigned bits) const {
        if (__any_sync(0xffffffffu, bits & 1u) && lane_id() == 0) set_flag(st, F_NAMES_DIFFER);
        if (__any_sync(0xffffffffu, bits & 2u) && lane_id() == 0) set_err(st, ERR_INVALID);
    }
};

// Name ids of every kernel below 2^24 (per-stream rows with layer classes,
// where the pairing above sees the replayed kernels only).
__global__ void k_check_names24(const uint32_t *__restrict__ name, int64_t n, DevStatus *st) {
    pdl_wait();
    uint32_t acc = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        acc |= name[i];
    if (__any_sync(0xffffffffu, acc >> 24 != 0) && lane_id() == 0) set_err(st, ERR_INVALID);
}

// ------------------------------------------------------------------ general path helpers
// Flags in time order: flag[i] = predicate(korder[i]).
//   what = 0: replayed (layer < 0 or the layer is its class representative)
//   what = 1: layer-tagged (layer >= 0)
__global__ void k_flags(const uint32_t *__restrict__ korder, const int32_t *__restrict__ layer,
                        const int32_t *__restrict__ rep_layer, int64_t n, int what, uint32_t *__restrict__ flag) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t k = korder ? korder[i] : i;
        int32_t l = layer ? layer[k] : -1;
        uint32_t f = what == 0 ? (l < 0 || rep_layer[l] == l) : (l >= 0);
        flag[i] = f;
    }
}
// Compact: list[pos[i]] = korder[i] where flag[i]
__global__ void k_compact(const uint32_t *__restrict__ korder, const uint32_t *__restrict__ flag,
                          const uint32_t *__restrict__ pos, int64_t n, uint32_t *__restrict__ list) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (flag[i]) list[pos[i]] = korder ? korder[i] : (uint32_t)i;
}
__global__ void k_gather_i32_as_u32(const int32_t *__restrict__ src, const uint32_t *__restrict__ idx, int64_t n,
                                    uint32_t *__restrict__ dst) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (uint32_t)src[idx[i]];
}
// The largest matching key (name, or name << 8 | stream with streams) of
// kernels and rows.
__global__ void k_max_key(const uint32_t *__restrict__ kname, const uint8_t *__restrict__ kstream, int64_t K,
                          const uint32_t *__restrict__ nname, const uint8_t *__restrict__ nstream, int64_t M,
                          DevStatus *st) {
    pdl_wait();
    uint32_t m = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < K + M; i += (int64_t)gridDim.x * blockDim.x) {
        const bool row = i >= K;
        const int64_t j = row ? i - K : i;
        uint32_t x = row ? nname[j] : kname[j];
        if (nstream) x = x << 8 | (row ? nstream[j] : kstream[j]);
        m = x > m ? x : m;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane_id() == 0 && m) atomicMax(&st->cnt[C_MAX_KEY], (unsigned long long)m);
}
__global__ void k_check_layers(const int32_t *__restrict__ layer, int64_t n, int32_t n_layers,
                               const int32_t *__restrict__ rep_layer, DevStatus *st) {
    pdl_wait();
    unsigned long long rep = 0;
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int32_t l = layer[i];
        if (l < -1 || l >= n_layers) bad = 1;
        else rep += (l < 0 || rep_layer[l] == l);
    }
    __shared__ unsigned long long red[33];
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_err(st, ERR_INVALID);
    block_add_u64(rep, &st->cnt[C_REPLAYED], red);
}

__device__ __forceinline__ int64_t lower_bound_u32(const uint32_t *a, int64_t n, uint32_t x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t m = (lo + hi) >> 1;
        if (a[m] < x) lo = m + 1; else hi = m;
    }
    return lo;
}
__device__ __forceinline__ int64_t upper_bound_u32(const uint32_t *a, int64_t n, uint32_t x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        int64_t m = (lo + hi) >> 1;
        if (a[m] <= x) lo = m + 1; else hi = m;
    }
    return lo;
}

// The sort's input: matching keys of the nrep replayed kernels in time order
// (list rk, or the kernel array itself when rk is null), then of the M rows.
// With streams the key is name << 8 | stream; a name id of 2^24 or more cannot
// be packed and is an invalid argument.
__global__ void k_pair_keys(const uint32_t *__restrict__ rk, const uint32_t *__restrict__ kname,
                            const uint8_t *__restrict__ kstream, int64_t nrep, const uint32_t *__restrict__ nname,
                            const uint8_t *__restrict__ nstream, int64_t n, uint32_t *__restrict__ key,
                            uint32_t *chain, int64_t nchain, DevStatus *st) {
    pdl_wait();
    zero_words(chain, nchain);               // of the runs' scan
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool row = i >= nrep;
        const int64_t j = row ? i - nrep : (rk ? (int64_t)rk[i] : i);
        uint32_t x = row ? nname[j] : kname[j];
        if (nstream) {
            bad |= x >> 24 != 0;
            x = x << 8 | (row ? nstream[j] : kstream[j]);
        }
        key[i] = x;
    }
    if (bad) set_err(st, ERR_INVALID);
}

// Runs of the sorted keys sk (sv[i] < nrep: a kernel, else a row): a name's
// kernels are one run, its rows the next.  run[i] is element i's run, start[u]
// the first element of run u; *n_run their number, start[*n_run] = n.
__device__ __forceinline__ bool run_head(const uint32_t *sk, const uint32_t *sv, int64_t nrep, int64_t i) {
    return i == 0 || sk[i - 1] != sk[i] || ((int64_t)sv[i - 1] < nrep) != ((int64_t)sv[i] < nrep);
}
__global__ void __launch_bounds__(SCAN_THREADS) k_runs(const uint32_t *__restrict__ sk,
                                                       const uint32_t *__restrict__ sv, int64_t nrep, int64_t n,
                                                       Chain C, uint32_t *__restrict__ run,
                                                       uint32_t *__restrict__ start, uint32_t *__restrict__ n_run) {
    pdl_wait();
    chained_scan(
        C, n, [&](int64_t i) -> uint32_t { return run_head(sk, sv, nrep, i); },
        [&](int64_t i, uint32_t head, uint32_t ex) {
            const uint32_t u = ex + head - 1;
            run[i] = u;
            if (head) start[u] = (uint32_t)i;
        },
        [&](uint32_t total) {
            *n_run = total;
            start[total] = (uint32_t)n;
        });
}

// The ordinal join over the sorted elements.  A kernel is the o-th of its name,
// o = i - start of its run; its row is the o-th element of the next run when
// that holds the name's rows, subject to the mismatch mode.  The first element
// of a kernel run compares its name's counts, the first of a row run reports a
// name without kernels.
__global__ void k_ordinal_join(const uint32_t *__restrict__ sk, const uint32_t *__restrict__ sv, int64_t nrep,
                               int64_t n, const uint32_t *__restrict__ run, const uint32_t *__restrict__ start,
                               const uint32_t *__restrict__ n_run, const uint32_t *__restrict__ rk, int mode,
                               int32_t *__restrict__ out_idx, uint8_t *__restrict__ out_kind, DevStatus *st) {
    pdl_wait();
    const uint32_t U = *n_run;
    unsigned long long direct = 0, unmatched = 0, names = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t j = sv[i], u = run[i], lo = start[u];
        if ((int64_t)j >= nrep) {
            names += lo == i && (i == 0 || sk[i - 1] != sk[i]);
            continue;
        }
        const uint32_t hi = start[u + 1];
        const bool rows = u + 1 < U && sk[hi] == sk[i];
        const uint32_t cq = rows ? start[u + 2] - hi : 0u, o = (uint32_t)i - lo;
        names += lo == i && hi - lo != cq;
        const bool ok = o < cq && (mode != OPATTR_MISMATCH_SKIP_NAME || hi - lo == cq);
        const int32_t idx = ok ? (int32_t)((int64_t)sv[hi + o] - nrep) : -1;
        const uint32_t k = rk ? rk[j] : j;
        out_idx[k] = idx;
        if (out_kind) out_kind[k] = idx >= 0 ? 1 : 0;
        direct += idx >= 0;
        unmatched += idx < 0;
    }
    __shared__ unsigned long long red[33];
    if (__any_sync(0xffffffffu, names != 0) && lane_id() == 0 && mode == OPATTR_MISMATCH_ERROR) set_err(st, ERR_COUNT);
    block_add_u64(direct, &st->cnt[C_DIRECT], red);
    block_add_u64(unmatched, &st->cnt[C_COUNT_UNMATCHED], red);
    block_add_u64(names, &st->cnt[C_NAMES_MISMATCH], red);
}

// ------------------------------------------------------------------ layers
// Layer deduplication with the kernels in time order, in one pass: each
// replayed kernel's rank among them is its row when the names agree and the
// rows are as many.  Layer ids are checked along the way.
__global__ void __launch_bounds__(SCAN_THREADS) k_layer_pairs(const int32_t *__restrict__ layer,
                                                              const int32_t *__restrict__ rep_layer, int32_t n_layers,
                                                              const uint32_t *__restrict__ kname,
                                                              const uint32_t *__restrict__ nname, int64_t K, int64_t M,
                                                              Chain C, int32_t *__restrict__ out_idx,
                                                              uint8_t *__restrict__ out_kind, DevStatus *st) {
    pdl_wait();
    int bad = 0, differ = 0;
    chained_scan(
        C, K,
        [&](int64_t i) -> uint32_t {
            const int32_t l = layer[i];
            const bool ok = l >= -1 && l < n_layers;
            bad |= !ok;
            return l < 0 || (ok && rep_layer[l] == l);
        },
        [&](int64_t i, uint32_t replayed, uint32_t rank) {
            if (!replayed) return;
            const bool row = (int64_t)rank < M;
            differ |= !row || kname[i] != nname[rank];
            out_idx[i] = row ? (int32_t)rank : -1;
            if (out_kind) out_kind[i] = 1;
        },
        [&](uint32_t total) {
            st->cnt[C_REPLAYED] = total;
            if ((int64_t)total != M) set_flag(st, F_NAMES_DIFFER);
        });
    if (bad) set_err(st, ERR_INVALID);
    if (differ) set_flag(st, F_NAMES_DIFFER);
}

// Positions within layers, few layers: one stable counting pass over the
// kernels in time order by layer id.
constexpr int LAYERS_DIGIT = RADIX_BINS - 1;        // with a last, empty digit for the end of the layer before
// (ids past the table are left out: this runs before the host has seen the check
// of the ids, and only the table's digits, and the empty one after them, have offsets)
struct LayerDigit {
    const int32_t *layer;
    const uint32_t *korder;
    int32_t n_layers;            // LAYERS_DIGIT at most
    __device__ __forceinline__ unsigned operator()(int64_t i) const {
        const int32_t l = layer[korder ? korder[i] : (uint32_t)i];
        return l >= 0 && l < n_layers ? (unsigned)l : (unsigned)RADIX_BINS;
    }
};
struct PlaceByLayer {
    const uint32_t *korder;
    uint32_t *list, *place;      // kernels layer by layer; each kernel's place there
    __device__ __forceinline__ unsigned operator()(int64_t i, uint32_t dest, unsigned) const {
        const uint32_t k = korder ? korder[i] : (uint32_t)i;
        list[dest] = k;
        place[k] = dest;
        return 0u;
    }
    __device__ __forceinline__ void done(unsigned) const {}
};
// offs[l * ntiles] is the first place of layer l.
__global__ void k_layer_broadcast(const int32_t *__restrict__ layer, const int32_t *__restrict__ rep_layer,
                                  int32_t n_layers, const uint32_t *__restrict__ offs, int64_t ntiles,
                                  const uint32_t *__restrict__ list, const uint32_t *__restrict__ place,
                                  const uint32_t *__restrict__ kname, int64_t K, int32_t *__restrict__ out_idx,
                                  uint8_t *__restrict__ out_kind, DevStatus *st) {
    pdl_wait();
    unsigned long long bc = 0, miss = 0;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < K; k += (int64_t)gridDim.x * blockDim.x) {
        const int32_t l = layer[k];
        if (l < 0 || l >= n_layers || rep_layer[l] == l) continue;
        const int32_t r = rep_layer[l];
        const uint32_t p = place[k] - offs[(int64_t)l * ntiles], r0 = offs[(int64_t)r * ntiles];
        int32_t idx = -1;
        if (p < offs[(int64_t)(r + 1) * ntiles] - r0) {
            const uint32_t src = list[r0 + p];
            if (kname[src] == kname[k]) idx = out_idx[src];
        }
        out_idx[k] = idx;
        if (out_kind) out_kind[k] = idx >= 0 ? 2 : 0;
        bc += idx >= 0;
        miss += idx < 0;
    }
    __shared__ unsigned long long red[33];
    block_add_u64(bc, &st->cnt[C_BROADCAST], red);
    block_add_u64(miss, &st->cnt[C_DEDUP_MISMATCH], red);
}

// Broadcast.  i runs over layer-tagged kernels sorted by (layer, time).
//   sll / slj: sorted layer ids and the time rank j of each (lk[j] = kernel)
__global__ void k_dedup_broadcast(const uint32_t *__restrict__ sll, const uint32_t *__restrict__ slj,
                                  const uint32_t *__restrict__ lk, int64_t nl, const int32_t *__restrict__ rep_layer,
                                  const uint32_t *__restrict__ kname, int32_t *__restrict__ out_idx,
                                  uint8_t *__restrict__ out_kind, DevStatus *st) {
    pdl_wait();
    unsigned long long bc = 0, miss = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nl; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t L = sll[i];
        int32_t rep = rep_layer[L];
        if ((uint32_t)rep == L) continue;                        // the representative itself: replayed
        int64_t lo = (i == 0 || sll[i - 1] != L) ? i : lower_bound_u32(sll, nl, L);
        int64_t p = i - lo;
        int64_t rlo = lower_bound_u32(sll, nl, (uint32_t)rep);
        int64_t rn = upper_bound_u32(sll, nl, (uint32_t)rep) - rlo;
        uint32_t k = lk[slj[i]];
        int32_t idx = -1;
        if (p < rn) {
            uint32_t src = lk[slj[rlo + p]];
            if (kname[src] == kname[k]) idx = out_idx[src];
        }
        out_idx[k] = idx;
        if (out_kind) out_kind[k] = idx >= 0 ? 2 : 0;
        bc += idx >= 0;
        miss += idx < 0;
    }
    __shared__ unsigned long long red[33];
    block_add_u64(bc, &st->cnt[C_BROADCAST], red);
    block_add_u64(miss, &st->cnt[C_DEDUP_MISMATCH], red);
}

// ------------------------------------------------------------------ host
static opattr_status read_u64(Ctx &c, const unsigned long long *d, unsigned long long *h) {
    if (cudaMemcpyAsync(h, d, sizeof(*h), cudaMemcpyDeviceToHost, c.stream) != cudaSuccess ||
        cudaStreamSynchronize(c.stream) != cudaSuccess)
        return cuda_status(c, cudaGetLastError());
    return OPATTR_OK;
}

// The stream-partitioned pairing over n replayed kernels (list rk, or the
// kernel array itself when rk is null) and the n rows.  Scratch: nb (n
// bytes), nv0 / nv1 (n).
static void stream_pairs(Ctx &c, const opattr_kernels *kern, const opattr_ncu *ncu, const uint32_t *rk, int64_t n,
                         uint8_t *nb, uint32_t *nv0, uint32_t *nv1, uint32_t *hist, uint32_t *part, int32_t *out_idx,
                         uint8_t *out_kind) {
    // rows: one 8-bit radix pass (it only reads the row streams)
    uint8_t *ko;
    uint32_t *pn;
    radix_sort_pairs<uint8_t>(c, const_cast<uint8_t *>(ncu->stream), nv0, nb, nv1, n, 8, true, hist, part, &ko, &pn);
    // kernels: ranked by stream, each paired in the same pass
    const StreamDigit dg{rk, kern->stream};
    const uint32_t *offs = digit_offsets(c, dg, n, hist, part);
    const StreamPairs ep{rk, pn, kern->name_id, ncu->name_id, kern->stream, ncu->stream, out_idx, out_kind,
                         c.d_status};
    digit_rank(c, "match_stream_pairs", dg, n, offs, ep);
}

bool match_layers_ahead(const opattr_dedup *dd) { return dd->n_layers > 0 && dd->n_layers <= LAYERS_DIGIT; }

// Every duplicate-layer kernel takes its representative's row.  Few layers:
// place / list from one counting pass; else layer-tagged kernels compacted in
// time order and sorted by layer.  korder: time order, or NULL.
static opattr_status broadcast_layers(Ctx &c, const opattr_kernels *kern, const opattr_dedup *dd, const int32_t *d_rep,
                                      const uint32_t *korder, uint32_t *flag, uint32_t *pos, uint32_t *lk,
                                      uint32_t *const *sort, uint32_t *hist, uint32_t *part, unsigned long long *dsm,
                                      int32_t *out_idx, uint8_t *out_kind) {
    const int64_t K = kern->n;
    const unsigned gK = grid_for(K, 256, REDUCE_GRID);
    if (dd->n_layers <= LAYERS_DIGIT) {
        const LayerDigit dg{kern->layer_id, korder, dd->n_layers};
        const uint32_t *offs = digit_offsets(c, dg, K, hist, part, dd->n_layers + 1);
        digit_rank(c, "layer_place", dg, K, offs, PlaceByLayer{korder, lk, pos});
        launch(c, "layer_broadcast", k_layer_broadcast, dim3(gK), dim3(256), 0, kern->layer_id, d_rep, dd->n_layers,
               offs, (K + RADIX_TILE - 1) / RADIX_TILE, (const uint32_t *)lk, (const uint32_t *)pos, kern->name_id, K,
               out_idx, out_kind, c.d_status);      // plain names: a class may span streams
        return OPATTR_OK;
    }
    launch(c, "flags", k_flags, dim3(gK), dim3(256), 0, korder, kern->layer_id, d_rep, K, 1, flag);
    uint32_t *ntag = reinterpret_cast<uint32_t *>(dsm + 1);
    scan_exclusive_u32(c, flag, pos, K, part, ntag);
    launch(c, "compact", k_compact, dim3(gK), dim3(256), 0, korder, (const uint32_t *)flag, (const uint32_t *)pos, K,
           lk);
    unsigned long long ntag_h = 0;
    const opattr_status st = read_u64(c, dsm + 1, &ntag_h);
    if (st) return st;
    const int64_t nlk = (int64_t)(ntag_h & 0xFFFFFFFFull);
    if (nlk == 0) return OPATTR_OK;
    launch(c, "gather_layers", k_gather_i32_as_u32, dim3(grid_for(nlk, 256, REDUCE_GRID)), dim3(256), 0,
           kern->layer_id, (const uint32_t *)lk, nlk, sort[0]);
    uint32_t *sll, *slj;
    radix_sort_pairs<uint32_t>(c, sort[0], sort[1], sort[2], sort[3], nlk,
                               bits_for((uint64_t)(dd->n_layers > 0 ? dd->n_layers - 1 : 0)), true, hist, part, &sll,
                               &slj);
    launch(c, "dedup_broadcast", k_dedup_broadcast, dim3(grid_for(nlk, 256, REDUCE_GRID)), dim3(256), 0,
           (const uint32_t *)sll, (const uint32_t *)slj, (const uint32_t *)lk, nlk, d_rep, kern->name_id, out_idx,
           out_kind, c.d_status);
    return OPATTR_OK;
}

opattr_status match_verdict(Ctx &c, opattr_match_summary *sum) {
    const DevStatus &H = *c.h_status;
    opattr_match_summary &S = c.match_sum;
    c.match_pending = false;
    if (H.err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
    if (H.err & ERR_COUNT) return OPATTR_E_COUNT_MISMATCH;
    if (S.replayed < 0) S.replayed = (int64_t)H.cnt[C_REPLAYED];     // layer pairs: counted on the way
    S.direct = S.fast_path ? S.replayed : (int64_t)H.cnt[C_DIRECT];
    S.broadcast = (int64_t)H.cnt[C_BROADCAST];
    S.names_mismatched = (int64_t)H.cnt[C_NAMES_MISMATCH];
    S.count_unmatched = S.fast_path ? 0 : (int64_t)H.cnt[C_COUNT_UNMATCHED];
    S.dedup_mismatch = (int64_t)H.cnt[C_DEDUP_MISMATCH];
    S.unmatched = S.kernels - S.direct - S.broadcast;
    if (sum) *sum = S;
    const int mode = (int)c.cfg.mismatch;
    if (mode == OPATTR_MISMATCH_SKIP_NAME && S.names_mismatched > 0) return OPATTR_W_COUNT_MISMATCH;
    if (mode == OPATTR_MISMATCH_PREFIX && S.count_unmatched > 0) return OPATTR_W_COUNT_MISMATCH;
    if (S.dedup_mismatch > 0) return OPATTR_W_DEDUP_MISMATCH;
    return OPATTR_OK;
}

// Scratch: the sort of kernels and rows (keys and values twice; the free pair then
// holds the runs), the time order, and with layers the replayed kernels and the
// layer lists.
struct MatchSizes {
    int64_t NL, N, NX, LX, hist_n, part_n;
    size_t bytes;
    MatchSizes(int64_t K, int64_t M, bool dedup_on, int64_t n_layers) {
        NL = dedup_on && n_layers > 0 ? n_layers : 1;
        N = K + M;
        NX = std::max(K, M);
        LX = dedup_on ? K : 1;
        hist_n = std::max(radix_hist_elems(N), radix_hist_elems(NX));
        part_n = scan_scratch_elems(std::max(std::max(hist_n, N), K));
        Need nd;
        nd.add<int32_t>(NL).add<unsigned long long>(4);
        for (int i = 0; i < 4; ++i) nd.add<uint32_t>(N + 2).add<uint32_t>(LX);
        nd.add<uint8_t>(NX).add<uint32_t>(hist_n).add<uint32_t>(part_n);
        bytes = nd.bytes + time_sort_scratch(K) + 4096;
    }
};
size_t match_scratch(int64_t K, int64_t M, bool dedup_on, int64_t n_layers) {
    return MatchSizes(K, M, dedup_on, n_layers).bytes;
}

opattr_status do_match(Ctx &c, const opattr_kernels *kern, const opattr_ncu *ncu, const opattr_dedup *dd,
                       int32_t *out_idx, uint8_t *out_kind, opattr_match_summary *sum) {
    const int64_t K = kern->n, M = ncu->n;
    c.rows_identity = false;
    if (K < 0 || M < 0 || K >= (1ll << 31) || M >= (1ll << 31)) return OPATTR_E_INVALID_ARG;
    if (K > 0 && (!kern->stream || !kern->start_ns || !kern->name_id || !out_idx)) return OPATTR_E_INVALID_ARG;
    if (M > 0 && !ncu->name_id) return OPATTR_E_INVALID_ARG;
    const int mode = (int)c.cfg.mismatch;
    const bool dedup_on = c.cfg.dedup && dd && kern->layer_id;
    std::vector<int32_t> rep_layer;
    if (dedup_on) {
        if (dd->n_layers < 0 || dd->n_classes < 0 || (dd->n_layers > 0 && !dd->class_of_layer) ||
            (dd->n_classes > 0 && !dd->rep_of_class))
            return OPATTR_E_INVALID_ARG;
        for (int32_t l = 0; l < dd->n_layers; ++l)
            if (dd->class_of_layer[l] < 0 || dd->class_of_layer[l] >= dd->n_classes) return OPATTR_E_INVALID_ARG;
        for (int32_t q = 0; q < dd->n_classes; ++q) {
            int32_t r = dd->rep_of_class[q];
            if (r < 0 || r >= dd->n_layers || dd->class_of_layer[r] != q) return OPATTR_E_INVALID_ARG;
        }
        rep_layer.resize(dd->n_layers > 0 ? dd->n_layers : 1);
        for (int32_t l = 0; l < dd->n_layers; ++l) rep_layer[l] = dd->rep_of_class[dd->class_of_layer[l]];
    }
    const bool per_stream = ncu->stream != nullptr;
    opattr_match_summary &S = c.match_sum;
    S = opattr_match_summary{};
    S.kernels = K;
    S.replayed = K;
    // within a join the identity pairing ran within the enclosure: with the
    // kernels in time order (the enclosure's verdict) and every name equal,
    // its outputs are the match
    // (with the enclosure's status still to be read, the names are taken to
    // agree; the join checks that verdict with the aggregation's status)
    if (c.spec_ran && c.order_from_enclose && c.enclose_k_sorted == 1 && c.spec_kname == kern->name_id &&
        c.spec_nname == ncu->name_id && c.spec_idx == out_idx &&
        c.spec_kind == out_kind && c.spec_k == K && K == M && !dedup_on && !per_stream &&
        (c.enclose_pending || !(c.h_status->flags & F_NAMES_DIFFER))) {
        S.direct = K;
        S.fast_path = 1;
        if (sum) *sum = S;
        c.rows_identity = true;
        return OPATTR_OK;
    }
    const MatchSizes Z(K, M, dedup_on, dedup_on ? dd->n_layers : 0);
    const int64_t NL = Z.NL, N = Z.N, NX = Z.NX, LX = Z.LX, hist_n = Z.hist_n, part_n = Z.part_n;
    opattr_status st = ensure_arena(c, Z.bytes);
    if (st) return st;
    Arena a(c);
    int32_t *d_rep = a.take<int32_t>(NL);
    unsigned long long *dsm = a.take<unsigned long long>(4);
    uint32_t *b0 = a.take<uint32_t>(N + 2), *b1 = a.take<uint32_t>(N + 2), *b2 = a.take<uint32_t>(N + 2),
             *b3 = a.take<uint32_t>(N + 2);
    uint32_t *flag = a.take<uint32_t>(LX), *pos = a.take<uint32_t>(LX), *rkb = a.take<uint32_t>(LX),
             *lk = a.take<uint32_t>(LX);
    uint8_t *nb = a.take<uint8_t>(NX);
    uint32_t *hist = a.take<uint32_t>(hist_n), *part = a.take<uint32_t>(part_n);
    if (!d_rep || !dsm || !b0 || !b1 || !b2 || !b3 || !flag || !pos || !rkb || !lk || !nb || !hist || !part)
        return OPATTR_E_OOM;
    // (nothing else uses the staging now: the enclosure before it in a join is
    // through with it once its status was read, or never used it)
    if (dedup_on && dd->n_layers > 0) {
        const size_t bytes = sizeof(int32_t) * dd->n_layers;
        if (bytes <= STAGE_BYTES && c.host_mapped) {
            memcpy(c.h_stage, rep_layer.data(), bytes);
            if ((st = copy_small(c, d_rep, c.h_stage, bytes, cudaMemcpyHostToDevice))) return st;
        } else {
            cudaMemcpyAsync(d_rep, rep_layer.data(), bytes, cudaMemcpyHostToDevice, c.stream);
        }
    }
    const unsigned gK = grid_for(K, 256, REDUCE_GRID);
    uint32_t *const sort[4] = {b0, b1, b2, b3};
    const bool few_layers = dedup_on && match_layers_ahead(dd);

    // within a join the enclosure has just verified these records' order (or its
    // verdict is pending and they are taken to be in order), and kept their time
    // order when they were out of it
    const bool known_sorted = c.order_from_enclose && c.enclose_k_sorted == 1;
    const bool known_unsorted = c.order_from_enclose && c.enclose_k_sorted == 0 && c.join_korder;
    // Fast paths, taking the kernel array to be in time order (confirmed or
    // refuted by the order check in the same batch, or by the join).
    const bool ahead = K > 0 && !known_unsorted && !c.no_spec;
    const bool try_identity = ahead && !dedup_on && !per_stream && K == M;
    const bool try_streams = ahead && !dedup_on && per_stream && K == M;
    const bool try_layers = ahead && few_layers && !per_stream;
    // with the enclosure's verdict pending the status block is its, and so is
    // the one that found the largest key; what the fast path finds is read with
    // the aggregation's status
    const bool defer = known_sorted && c.enclose_pending && (try_streams || try_layers);
    const bool sort_at_once = known_sorted && !dedup_on && c.max_known && !c.enclose_pending && !try_identity &&
                              !try_streams;
    // kernels that the enclosure found out of order, as many rows: the pairing
    // through the time order comes first, on the clear status it left
    const bool list_at_once = known_unsorted && !dedup_on && K == M && !c.no_spec;
    const bool at_once = sort_at_once || list_at_once;
    const ZeroRun zc{part, chain_words(K)};
    uint64_t max_key = 0;
    if (defer) {
        if (try_layers && (st = zero_runs(c, 1, &zc))) return st;
    } else if (at_once) {
        if (sort_at_once) max_key = c.h_status->cnt[C_MAX_KEY];
    } else if ((st = reset_status(c, try_layers ? 1 : 0, &zc))) {
        return st;
    }
    if (!at_once) {
        if (!known_sorted && !known_unsorted) check_kernel_order(c, kern->stream, kern->start_ns, K);
        if (try_layers)
            launch(c, "layer_pairs", k_layer_pairs, dim3(grid_for(K, SCAN_TILE)), dim3(SCAN_THREADS), 0,
                   kern->layer_id, (const int32_t *)d_rep, dd->n_layers, kern->name_id, ncu->name_id, K, M,
                   make_chain(c, part, K), out_idx, out_kind, c.d_status);
        else if (dedup_on && K > 0)
            launch(c, "check_layers", k_check_layers, dim3(gK), dim3(256), 0, kern->layer_id, K, dd->n_layers,
                   (const int32_t *)d_rep, c.d_status);
        if (per_stream && dedup_on && K > 0)
            launch(c, "check_names24", k_check_names24, dim3(grid_for(K, 256 * 8, REDUCE_GRID)), dim3(256), 0,
                   kern->name_id, K, c.d_status);
        if (try_identity)
            launch(c, "match_identity", k_match_identity, dim3(grid_for(K, 256 * 16, REDUCE_GRID)), dim3(256), 0,
                   kern->name_id, ncu->name_id, K, out_idx, out_kind,
                   identity_vec(kern->name_id, ncu->name_id, out_idx, out_kind), c.d_status);
        if (try_streams) stream_pairs(c, kern, ncu, nullptr, K, nb, b0, b1, hist, part, out_idx, out_kind);
        if (try_layers && (st = broadcast_layers(c, kern, dd, d_rep, nullptr, flag, pos, lk, sort, hist, part, dsm,
                                                 out_idx, out_kind)))
            return st;
        // (a pairing that is tried before the sort, here or below, rarely fails:
        // the largest key is then found afterwards)
        if (!defer && N > 0 && !try_identity && !try_streams && !try_layers && (!dedup_on || c.no_spec))
            launch(c, "max_key", k_max_key, dim3(grid_for(N, 256 * 8, 1024)), dim3(256), 0, kern->name_id, kern->stream,
                   K, ncu->name_id, ncu->stream, M, c.d_status);
        if (defer) {
            S.fast_path = 1;
            if (try_layers) S.replayed = -1;
            c.match_pending = true;
            return OPATTR_OK;
        }
        if ((st = read_status(c))) return st;
        if (c.h_status->err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
        max_key = c.h_status->cnt[C_MAX_KEY];
        const bool sorted = known_sorted || (!known_unsorted && !(c.h_status->flags & F_K_UNSORTED));
        if (dedup_on) S.replayed = (int64_t)c.h_status->cnt[C_REPLAYED];
        if ((try_identity || try_streams || try_layers) && sorted && !(c.h_status->flags & F_NAMES_DIFFER)) {
            S.fast_path = 1;
            return match_verdict(c, sum);
        }
        // the speculative verdicts are spent: later checks start from clear flags and counts
        const ZeroRun zr[2] = {{&c.d_status->flags, 1}, {&c.d_status->cnt[0], 2 * C_MAX_KEY}};
        if ((st = zero_runs(c, 2, zr))) return st;
    }
    const bool k_sorted = known_sorted || (!known_unsorted && !(c.h_status->flags & F_K_UNSORTED));

    // ---- general path
    uint32_t *korder = nullptr;
    if (!k_sorted && K > 0) {
        if (known_unsorted) korder = c.join_korder;
        else if ((st = kernel_time_order(c, a, kern->stream, kern->start_ns, K, &korder))) return st;
    }
    // rk[j] = kernel index of the j-th replayed kernel in time order (NULL: j itself)
    int64_t nrep = K;
    const uint32_t *rk = korder;
    if (dedup_on && K > 0) {
        launch(c, "flags", k_flags, dim3(gK), dim3(256), 0, (const uint32_t *)korder, kern->layer_id,
               (const int32_t *)d_rep, K, 0, flag);
        scan_exclusive_u32(c, flag, pos, K, part, nullptr);
        launch(c, "compact", k_compact, dim3(gK), dim3(256), 0, (const uint32_t *)korder, (const uint32_t *)flag,
               (const uint32_t *)pos, K, rkb);
        nrep = S.replayed;
        rk = rkb;
        // (duplicate-layer kernels are written by the broadcast, the others by the join)
    }
    bool direct_done = false;
    // rows equal to the replayed kernels in time order, tried before the name
    // sort: with layer deduplication, or when the kernels were out of time order
    const bool retry_streams = per_stream && !c.no_spec && (dedup_on || korder) && nrep == M && nrep > 0;
    const bool retry_list = !per_stream && !c.no_spec && (korder || (dedup_on && !try_layers)) && nrep == M &&
                            nrep > 0;
    if (retry_streams || retry_list) {
        if (retry_streams) stream_pairs(c, kern, ncu, rk, nrep, nb, b0, b1, hist, part, out_idx, out_kind);
        else
            launch(c, "match_identity_list", k_match_identity_list, dim3(grid_for(nrep, 256, REDUCE_GRID)),
                   dim3(256), 0, rk, kern->name_id, ncu->name_id, nrep, out_idx, out_kind, c.d_status);
        if ((st = read_status(c))) return st;
        if (c.h_status->err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
        direct_done = !(c.h_status->flags & F_NAMES_DIFFER);
    }
    if (!direct_done && (nrep > 0 || M > 0)) {
        const int64_t n = nrep + M;
        uint32_t *chain = reinterpret_cast<uint32_t *>(nb);          // free by now; two words per 4,096 elements fit
        if (max_key == 0) {
            launch(c, "max_key", k_max_key, dim3(grid_for(N, 256 * 8, 1024)), dim3(256), 0, kern->name_id, kern->stream,
                   K, ncu->name_id, ncu->stream, M, c.d_status);
            if ((st = read_status(c))) return st;
            max_key = c.h_status->cnt[C_MAX_KEY];
        }
        launch(c, "pair_keys", k_pair_keys, dim3(grid_for(n, 256 * 4, REDUCE_GRID)), dim3(256), 0, rk, kern->name_id,
               kern->stream, nrep, ncu->name_id, ncu->stream, n, b0, chain, chain_words(n), c.d_status);
        uint32_t *sk = nullptr, *sv = nullptr;
        radix_sort_pairs<uint32_t>(c, b0, b1, b2, b3, n, bits_for(max_key), true, hist, part, &sk, &sv);
        uint32_t *run = sk == b0 ? b2 : b0, *start = sv == b1 ? b3 : b1;
        uint32_t *n_run = reinterpret_cast<uint32_t *>(dsm + 2);
        launch(c, "runs", k_runs, dim3(grid_for(n, SCAN_TILE)), dim3(SCAN_THREADS), 0, (const uint32_t *)sk,
               (const uint32_t *)sv, nrep, n, make_chain(c, chain, n), run, start, n_run);
        launch(c, "ordinal_join", k_ordinal_join, dim3(grid_for(n, 256 * 2, REDUCE_GRID)), dim3(256), 0,
               (const uint32_t *)sk, (const uint32_t *)sv, nrep, n, (const uint32_t *)run, (const uint32_t *)start,
               (const uint32_t *)n_run, rk, mode, out_idx, out_kind, c.d_status);
    }
    S.fast_path = direct_done ? 1 : 0;
    if (dedup_on && K > 0 && (st = broadcast_layers(c, kern, dd, d_rep, korder, flag, pos, lk, sort, hist, part, dsm,
                                                    out_idx, out_kind)))
        return st;
    if (c.in_join) {
        // complete but for its counts, read with the aggregation's status
        c.match_pending = c.keep_status = true;
        return OPATTR_OK;
    }
    if ((st = read_status(c))) return st;
    return match_verdict(c, sum);
}

}  // namespace opattr
