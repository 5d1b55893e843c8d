// enclose.cu -- Algorithm 2 (NVTX enclosure attribution, Sec. 3.5) on the GPU.
//
// Kernels in time order and ranges in start order are walked together, as one
// merged sequence of events in which a range comes before the kernels that
// start no earlier.  The sequence is cut into tiles of equal length, runs of
// tiles into parts, one block each; a block needs, besides its own events, only
// the last range before it on every level (stream, depth), because within a
// level ranges are disjoint or touching, so "the last range with start <= T"
// is the only one that can contain T.  Three launches, no host decision
// between them:
//   enc_parts  checks kernel and range records (order, intervals, depths);
//              each tile's place in the merged sequence, and the last range of
//              every level inside each part
//   enc_carry  those, made a running maximum over the parts (many parts only)
//   enclose    the parts, tile by tile: parents, chains and laminar checks of
//              the tile's ranges in shared memory, then its kernels
// Nothing is regrouped in device memory: kernels and ranges are read where
// they lie, in order, and results are written in order.  Records out of order
// are found by enc_parts (the other two then leave at once), sorted, and the
// last two run again on the sorted view; so they do with wider tables, by groups of
// streams or with wider times where the levels, the streams or the times ask for it.
#include <algorithm>
#include <type_traits>

#include "sort.cuh"
#include "util.cuh"

namespace opattr {

constexpr int LEVELS = N_LEVELS;
constexpr uint32_t KIND_OP = 0, KIND_NONOP = 1, KIND_STRUCT = 2;
constexpr uint32_t POS_MASK = 0x3FFFFFFFu;

__device__ __forceinline__ uint32_t kind_of(uint32_t op) {
    return op == OPATTR_OP_STRUCTURAL ? KIND_STRUCT : (op == OPATTR_OP_NONOP ? KIND_NONOP : KIND_OP);
}

// Kernels in time order, ranges in start order: the caller's arrays, or the
// sorted view of records out of order (kernels as the sorted time keys,
// ranges as sorted copies; korder / perm give the caller's indices).
struct EncView {
    const int64_t *k_start;
    const uint8_t *k_stream;
    const uint64_t *k_key;       // (start - k_tmin) << k_sbits | compact stream id, or NULL
    long long k_tmin;
    int k_sbits;
    const uint8_t *k_unmap;      // stream of each compact id
    const uint32_t *korder;      // NULL = array order
    int64_t K;
    const int64_t *r_start, *r_end;
    const uint8_t *r_stream, *r_depth;
    const uint32_t *r_op;
    const uint32_t *perm;        // NULL = array order
    int64_t R;

    template <bool KEYS>
    __device__ __forceinline__ long long time(int64_t i) const {
        return KEYS ? k_tmin + (long long)(k_key[i] >> k_sbits) : k_start[i];
    }
    template <bool KEYS>
    __device__ __forceinline__ unsigned stream(int64_t i) const {
        return KEYS ? k_unmap[(unsigned)k_key[i] & ((1u << k_sbits) - 1u)] : k_stream[i];
    }
};

// ------------------------------------------------------------------ parts
// The merged events of tile i of n: [tile_event(i), tile_event(i + 1)).
// Part b of the tiles' parts is tiles [b * tp, (b + 1) * tp).
__device__ __forceinline__ int64_t tile_event(int64_t i, int64_t n, int64_t events) {
    return (int64_t)((unsigned long long)events * (unsigned long long)i / (unsigned long long)n);   // below 2^52
}

// Traces with more streams or levels than one block's tables hold are taken group
// by group of 16 consecutive stream ids (512 levels at most): kernels and ranges
// partitioned stably by group, every group a sequence of its own with a share of
// the parts in proportion to its events.  20M kernels, enclosure and partition:
// 255 streams of 12 levels 510 + 390 us, where four walks of the whole trace with the
// streams of one group each took 2,388; of 32 levels 690 + 395 and 2,805.
constexpr int GROUP_SHIFT = 4, N_GROUPS = 256 >> GROUP_SHIFT;
struct EncGroup {
    int64_t k0, K, r0, R, tile0;         // its kernels, ranges and tile bounds begin at
    int part0, parts, tp;
};
// View and parts narrowed to the group of part b; false for a block past the last part.
__device__ __forceinline__ bool enter_group(const EncGroup *__restrict__ G, EncView &V, int64_t &b, int64_t &parts, int &tp,
                                            int64_t &tile0, int64_t &part0, unsigned &grp) {
    unsigned g = 0;
    while (g < N_GROUPS && b >= G[g].part0 + G[g].parts) ++g;
    if (g == N_GROUPS) return false;
    const EncGroup E = G[g];
    V.k_start += E.k0;
    V.k_stream += E.k0;
    V.korder += E.k0;
    V.K = E.K;
    V.r_start += E.r0;
    V.r_end += E.r0;
    V.r_stream += E.r0;
    V.r_depth += E.r0;
    V.r_op += E.r0;
    V.perm += E.r0;
    V.R = E.R;
    b -= E.part0;
    parts = E.parts;
    tp = E.tp;
    tile0 = E.tile0;
    part0 = E.part0;
    grp = g;
    return true;
}

// Ranges among the first d[i] merged events for each i, by one warp: 32 probes
// a round, the N searches' side by side (a round is two gathers' latency).  A
// range precedes the kernels that start no earlier.  Ends in [0, R] whatever the
// order of the records.
template <bool KEYS, int N>
__device__ __forceinline__ void ranges_before(const EncView &V, const int64_t (&d)[N], int64_t (&lo)[N]) {
    const unsigned lane = lane_id();
    int64_t hi[N];
    bool more = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        lo[i] = d[i] > V.K ? d[i] - V.K : 0;
        hi[i] = d[i] < V.R ? d[i] : V.R;
        more |= lo[i] < hi[i];
    }
    while (more) {
        bool before[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int64_t p = lo[i] + (int64_t)lane * ((hi[i] - lo[i] + 31) >> 5);
            before[i] = p < hi[i] && V.r_start[p] <= V.time<KEYS>(d[i] - p - 1);
        }
        more = false;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const unsigned m = ~__ballot_sync(0xffffffffu, before[i]);
            const int64_t step = (hi[i] - lo[i] + 31) >> 5;
            const int c = m ? __ffs(m) - 1 : 32;      // lanes 0 .. c - 1 lie before
            if (c == 0) {
                hi[i] = lo[i];
                continue;
            }
            const int64_t nh = lo[i] + (int64_t)c * step;
            lo[i] += (int64_t)(c - 1) * step + 1;
            hi[i] = nh < hi[i] ? nh : hi[i];
            more |= lo[i] < hi[i];
        }
    }
}

// What enc_parts checks and, within a join, the matching's identity pairing
// (row j for kernel j), written in the same pass over the kernels.
struct EncCheck {
    const uint32_t *kname, *nname;       // NULL: no pairing
    int32_t *idx;
    uint8_t *kind;                       // may be NULL
    int vec;                             // kernel arrays aligned for 16-byte accesses
    int pair_vec;                        // the pairing's arrays too
    const uint32_t *mk, *mn;             // names of kernels and rows whose largest key is wanted, or NULL
    const uint8_t *ms;                   // streams of the rows: keys are name << 8 | stream
    int64_t M;
};

constexpr int EP_THREADS = 256;
constexpr int EP_G = 8;                  // consecutive kernels of a thread; ranges whose loads go together
constexpr int EP_SEARCH = 4;             // tile bounds a warp looks for at once
// One block per part of tp tiles.  With CHECK it also verifies an equal share of the
// records as they lie: kernel order (start, stream), range intervals, depths
// and start order, the smallest and largest times, the streams with kernels
// and the depths present on every stream.  Then the tiles' bounds in the
// merged sequence (tile_r: ranges before each tile) and, in shared memory, the
// last range of every level among the part's ranges, written as a row of `rows`
// up to the highest level present (row_len; position + 1, 0 for none).
//
// Bound by HBM: 9 bytes per kernel and 18 per range (13 more per kernel with
// the pairing), each read or written once: 121 us for 20M kernels and 5.1M
// ranges in order, 4.4 TB/s (130 with a tile bound and a range at a time).
template <bool CHECK, bool KEYS, bool GROUPS = false>
__global__ void __launch_bounds__(EP_THREADS) k_enc_parts(EncView V, EncCheck C, int64_t parts, int tp,
                                                          uint32_t *__restrict__ tile_r, uint32_t *__restrict__ rows,
                                                          uint32_t *__restrict__ row_len,
                                                          uint32_t *__restrict__ lvlmask, const EncGroup *__restrict__ G,
                                                          DevStatus *st) {
    pdl_wait();
    __shared__ uint32_t last[LEVELS];
    __shared__ uint32_t dmask[256];
    __shared__ uint8_t kseen[256];
    __shared__ int flags_s;
    __shared__ long long mm_s[4];
    __shared__ int64_t bound[2];
    __shared__ uint32_t top_s;
    const int tid = threadIdx.x;
    int64_t b = blockIdx.x;
    if (GROUPS) {
        int64_t tile0, part0;
        unsigned grp;
        if (!enter_group(G, V, b, parts, tp, tile0, part0, grp)) return;
        tile_r += tile0;
        rows += part0 * LEVELS;
        row_len += part0;
    }
    const unsigned lane = lane_id(), warp = tid >> 5;
    for (int i = tid; i < LEVELS; i += EP_THREADS) last[i] = 0;
    if (CHECK) {
        for (int i = tid; i < 256; i += EP_THREADS) {
            dmask[i] = 0;
            kseen[i] = 0;
        }
        if (tid == 0) {
            flags_s = 0;
            mm_s[0] = mm_s[2] = LLONG_MAX;
            mm_s[1] = mm_s[3] = LLONG_MIN;
        }
    }
    if (tid == 0) top_s = 0;
    __syncthreads();
    if (CHECK) {
        enum { U_KERN = 1, U_RANGE = 2, BAD_END = 4, BAD_DEPTH = 8, NAMES = 16 };
        int f = 0;
        long long kmn = LLONG_MAX, kmx = LLONG_MIN, rmn = LLONG_MAX, rmx = LLONG_MIN;
        const int64_t kshare = ((V.K + parts - 1) / parts + EP_G - 1) / EP_G * EP_G;
        const int64_t kb = b * kshare, ke = kb + kshare < V.K ? kb + kshare : V.K;
        for (int64_t i0 = kb + (int64_t)tid * EP_G; i0 < ke; i0 += EP_THREADS * EP_G) {
            long long t[EP_G + 1];
            unsigned s[EP_G + 1];
            const bool whole = i0 + EP_G <= V.K;
            if (C.vec && whole) {
                const longlong2 *p = reinterpret_cast<const longlong2 *>(V.k_start + i0);
#pragma unroll
                for (int q = 0; q < EP_G / 2; ++q) {
                    const longlong2 x = p[q];
                    t[2 * q] = x.x;
                    t[2 * q + 1] = x.y;
                }
                const uint2 w = *reinterpret_cast<const uint2 *>(V.k_stream + i0);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    s[u] = (w.x >> (8 * u)) & 0xFFu;
                    s[4 + u] = (w.y >> (8 * u)) & 0xFFu;
                }
            } else {
#pragma unroll
                for (int u = 0; u < EP_G; ++u) {
                    t[u] = i0 + u < V.K ? V.k_start[i0 + u] : LLONG_MAX;
                    s[u] = i0 + u < V.K ? V.k_stream[i0 + u] : 255u;
                }
            }
            t[EP_G] = i0 + EP_G < V.K ? V.k_start[i0 + EP_G] : LLONG_MAX;
            s[EP_G] = i0 + EP_G < V.K ? V.k_stream[i0 + EP_G] : 255u;
            if (C.kname) {
                if (C.pair_vec && whole) {
                    uint4 x[2], y[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        x[q] = *reinterpret_cast<const uint4 *>(C.kname + i0 + 4 * q);
                        y[q] = *reinterpret_cast<const uint4 *>(C.nname + i0 + 4 * q);
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        if ((x[q].x != y[q].x) | (x[q].y != y[q].y) | (x[q].z != y[q].z) | (x[q].w != y[q].w)) f |= NAMES;
                        const int32_t j = (int32_t)(i0 + 4 * q);
                        *reinterpret_cast<int4 *>(C.idx + j) = make_int4(j, j + 1, j + 2, j + 3);
                    }
                    if (C.kind) *reinterpret_cast<uint2 *>(C.kind + i0) = make_uint2(0x01010101u, 0x01010101u);
                } else {
                    for (int u = 0; u < EP_G && i0 + u < V.K; ++u) {
                        if (C.kname[i0 + u] != C.nname[i0 + u]) f |= NAMES;
                        C.idx[i0 + u] = (int32_t)(i0 + u);
                        if (C.kind) C.kind[i0 + u] = 1;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < EP_G; ++u) {
                if (i0 + u >= V.K) break;
                kmn = t[u] < kmn ? t[u] : kmn;
                kmx = t[u] > kmx ? t[u] : kmx;
                if (i0 + u + 1 < V.K && (t[u + 1] < t[u] || (t[u + 1] == t[u] && s[u + 1] < s[u]))) f |= U_KERN;
                kseen[s[u]] = 1;
            }
        }
        const int64_t rshare = (V.R + parts - 1) / parts;
        const int64_t rb = b * rshare, re = rb + rshare < V.R ? rb + rshare : V.R;
        constexpr int B = 4;             // ranges of a thread, loads issued together
        for (int64_t j0 = rb + tid; j0 < re; j0 += EP_THREADS * B) {
            long long sv[B], ev[B], nv[B];
            unsigned dv[B], tv[B];
#pragma unroll
            for (int u = 0; u < B; ++u) {
                const int64_t i = j0 + u * EP_THREADS;
                const bool in = i < re;
                sv[u] = in ? V.r_start[i] : 0;
                ev[u] = in ? V.r_end[i] : 0;
                nv[u] = in && i + 1 < V.R ? V.r_start[i + 1] : LLONG_MAX;
                dv[u] = in ? V.r_depth[i] : 0u;
                tv[u] = in ? V.r_stream[i] : 0u;
            }
#pragma unroll
            for (int u = 0; u < B; ++u) {
                if (j0 + u * EP_THREADS >= re) break;
                if (ev[u] < sv[u]) f |= BAD_END;
                if (dv[u] >= OPATTR_MAX_DEPTH) f |= BAD_DEPTH;
                if (nv[u] < sv[u]) f |= U_RANGE;
                rmn = sv[u] < rmn ? sv[u] : rmn;
                rmx = ev[u] > rmx ? ev[u] : rmx;
                if (dv[u] < OPATTR_MAX_DEPTH && !((dmask[tv[u]] >> dv[u]) & 1u)) atomicOr(&dmask[tv[u]], 1u << dv[u]);
            }
        }
        if (C.mk) {
            uint32_t top_key = 0;
            for (int64_t i = kb + tid; i < ke; i += EP_THREADS) {
                const uint32_t x = C.ms ? C.mk[i] << 8 | V.k_stream[i] : C.mk[i];
                top_key = x > top_key ? x : top_key;
            }
            const int64_t mshare = (C.M + parts - 1) / parts, me = (b + 1) * mshare < C.M ? (b + 1) * mshare : C.M;
            for (int64_t i = b * mshare + tid; i < me; i += EP_THREADS) {
                const uint32_t x = C.ms ? C.mn[i] << 8 | C.ms[i] : C.mn[i];
                top_key = x > top_key ? x : top_key;
            }
            top_key = __reduce_max_sync(0xffffffffu, top_key);
            if (lane == 0 && top_key) atomicMax(&st->cnt[C_MAX_KEY], (unsigned long long)top_key);
        }
        f = (int)__reduce_or_sync(0xffffffffu, (unsigned)f);
        if (lane == 0 && f) atomicOr(&flags_s, f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long a0 = __shfl_xor_sync(0xffffffffu, kmn, o), a1 = __shfl_xor_sync(0xffffffffu, kmx, o);
            const long long a2 = __shfl_xor_sync(0xffffffffu, rmn, o), a3 = __shfl_xor_sync(0xffffffffu, rmx, o);
            kmn = a0 < kmn ? a0 : kmn;
            kmx = a1 > kmx ? a1 : kmx;
            rmn = a2 < rmn ? a2 : rmn;
            rmx = a3 > rmx ? a3 : rmx;
        }
        if (lane == 0) {
            atomicMin(&mm_s[0], kmn);
            atomicMax(&mm_s[1], kmx);
            atomicMin(&mm_s[2], rmn);
            atomicMax(&mm_s[3], rmx);
        }
        __syncthreads();
        if (tid < 256) {
            const uint32_t m = dmask[tid];
            if (m) atomicOr(&lvlmask[tid], m);
            const unsigned w = __ballot_sync(0xffffffffu, kseen[tid] != 0);
            if (lane == 0 && w) atomicOr(&st->kstreams[warp], w);
        }
        if (tid == 0) {
            if (flags_s & BAD_END) set_err(st, ERR_INVALID);
            if (flags_s & BAD_DEPTH) set_err(st, ERR_DEPTH);
            const unsigned fl = ((flags_s & U_KERN) ? F_K_UNSORTED : 0u) | ((flags_s & U_RANGE) ? F_R_UNSORTED : 0u) |
                                ((flags_s & NAMES) ? F_NAMES_DIFFER : 0u);
            if (fl) set_flag(st, fl);
            if (kb < ke) {
                atomicMin(&st->mm[MM_KSTART_MIN], mm_s[0]);
                atomicMax(&st->mm[MM_KSTART_MAX], mm_s[1]);
            }
            if (rb < re) {
                atomicMin(&st->mm[MM_RSTART_MIN], mm_s[2]);
                atomicMax(&st->mm[MM_REND_MAX], mm_s[3]);
            }
        }
    }
    // the part's tiles and ranges
    const int64_t nt = parts * tp, t0 = b * tp;
    for (int q0 = (int)warp; q0 <= tp; q0 += EP_THREADS / 32 * EP_SEARCH) {
        int64_t d[EP_SEARCH], r[EP_SEARCH];
#pragma unroll
        for (int i = 0; i < EP_SEARCH; ++i) {
            const int q = q0 + i * (EP_THREADS / 32);
            d[i] = q <= tp ? tile_event(t0 + q, nt, V.K + V.R) : 0;
        }
        ranges_before<KEYS>(V, d, r);
        if (lane != 0) continue;
#pragma unroll
        for (int i = 0; i < EP_SEARCH; ++i) {
            const int q = q0 + i * (EP_THREADS / 32);
            if (q > tp) break;
            if (q < tp || t0 + q == nt) tile_r[t0 + q] = (uint32_t)r[i];
            if (q == 0) bound[0] = r[i];
            if (q == tp) bound[1] = r[i];
        }
    }
    __syncthreads();
    const int64_t r0 = bound[0];
    // (records out of order, whose bounds mean nothing: no more than a part's worth)
    const int64_t most = r0 + tile_event(t0 + tp, nt, V.K + V.R) - tile_event(t0, nt, V.K + V.R);
    const int64_t r1 = bound[1] < most ? bound[1] : most;
    uint32_t top = 0;
    for (int64_t i0 = r0 + tid; i0 < r1; i0 += EP_THREADS * EP_G) {
        unsigned dv[EP_G], sv[EP_G];
#pragma unroll
        for (int u = 0; u < EP_G; ++u) {
            const int64_t i = i0 + u * EP_THREADS;
            dv[u] = i < r1 ? V.r_depth[i] : (unsigned)OPATTR_MAX_DEPTH;
            sv[u] = i < r1 ? V.r_stream[i] : 0u;
        }
#pragma unroll
        for (int u = 0; u < EP_G; ++u) {
            if (dv[u] >= OPATTR_MAX_DEPTH) continue;
            const unsigned l = sv[u] * 32u + dv[u];
            atomicMax(&last[l], (uint32_t)(i0 + u * EP_THREADS) + 1u);
            top = l + 1 > top ? l + 1 : top;
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0 && top) atomicMax(&top_s, top);
    __syncthreads();
    const uint32_t n = top_s;
    for (uint32_t i = tid; i < n; i += EP_THREADS) rows[b * LEVELS + i] = last[i];
    if (tid == 0) row_len[b] = n;
}

// Rows of the parts' last ranges to rows of the last range before each part:
// a running maximum down every column.  One block per stream: lane d of a
// warp takes depth d, each of the 32 warps an equal run of the parts.
template <bool GROUPS>
__global__ void __launch_bounds__(1024) k_enc_carry(uint32_t *__restrict__ rows, const uint32_t *__restrict__ row_len,
                                                    int64_t parts, const uint32_t *__restrict__ lvlmask,
                                                    const EncGroup *__restrict__ G) {
    pdl_wait();
    if (lvlmask[blockIdx.x] == 0) return;
    if (GROUPS) {                                // the parts of the stream's group
        G += blockIdx.x >> GROUP_SHIFT;
        rows += (int64_t)G->part0 * LEVELS;
        row_len += G->part0;
        parts = G->parts;
    }
    __shared__ uint32_t seg[32][33];
    const unsigned lane = lane_id(), w = threadIdx.x >> 5;
    const uint32_t l = blockIdx.x * 32u + lane;
    const int64_t per = (parts + 31) / 32;
    const int64_t b0 = w * per, b1 = b0 + per < parts ? b0 + per : parts;
    uint32_t m = 0;
#pragma unroll 8
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t v = l < row_len[b] ? rows[b * LEVELS + l] : 0u;
        m = v > m ? v : m;
    }
    seg[w][lane] = m;
    __syncthreads();
    m = 0;
    for (unsigned q = 0; q < w; ++q) m = seg[q][lane] > m ? seg[q][lane] : m;
#pragma unroll 8
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t v = l < row_len[b] ? rows[b * LEVELS + l] : 0u;
        rows[b * LEVELS + l] = m;
        m = v > m ? v : m;
    }
}

// ------------------------------------------------------------------ enclosure
// Shared memory of a tile: entries 0 .. SR - 1 are its ranges in order, entry
// SR + l the range open on level l when the tile begins (alive bits in amask).
// Levels of a stream are consecutive, depth by depth; 16-bit indices name
// entries, E_NONE none.
constexpr unsigned E_NONE = 0xFFFFu;
constexpr unsigned D_DEPTH = 31u, D_MIXED = 32u;     // bits of `dep`
template <int THREADS_, int BLOCKS_, bool JUMP_, typename Time_>
struct EncTile {
    using Time = Time_;                              // of a step, relative to its first event
    static constexpr int THREADS = THREADS_, BLOCKS = BLOCKS_;
    static constexpr bool JUMP = JUMP_;
    static constexpr int WORDS = 16;                 // ranges of a step, 32 to a group
    static constexpr int SR = 32 * WORDS;
    static constexpr int RPT = WORDS / (THREADS / 32);   // groups of a warp
    Time *ss, *se;               // start, end (relative)
    uint32_t *si;                // position | kind << 30
    uint32_t *amask;             // [ns] depths with an open range, per compact stream
    uint32_t *smask;             // [ns][WORDS] the stream's ranges among the tile's, one bit each
    uint32_t *sgroups;           // [ns] the groups that hold some
    uint16_t *par, *prev, *best; // parent; the entry before on the stream; where the climb begins (below)
    uint16_t *va;                // innermost operator of the entry's chain
    uint16_t *top;               // outermost ancestor
    uint16_t *jump;              // with JUMP: ancestor four levels up, E_NONE none (where chains are long)
    uint16_t *before;            // [ns][WORDS] the stream's last entry before each group (before the first one
                                 // its deepest open range), E_NONE none
    uint32_t *lgroups;           // [nl / 2] the groups that hold ranges of a level, 16 bits each
    uint8_t *last;               // [WORDS][nl] last range of each level in such a group
    uint16_t *cbase;             // [256] first level of a stream
    uint16_t *scid;              // [256] compact id of a stream (streams with levels, in order), E_NONE none
    uint8_t *dep, *vn;           // depth | D_MIXED; operators in the chain
    uint8_t *sid;                // compact stream of the tile's ranges
    uint8_t *ndep;               // [256] levels of a stream
    uint8_t *slist;              // [256] the stream of a compact id
    uint8_t *tlist;              // [ns] the streams that have ranges in the tile
    __device__ __forceinline__ EncTile(unsigned char *p, int nl, int ns) {
        const int cap = SR + nl;
        auto take = [&](size_t n) { unsigned char *q = p; p += n; return q; };
        ss = reinterpret_cast<Time *>(take((size_t)cap * sizeof(Time)));
        se = reinterpret_cast<Time *>(take((size_t)cap * sizeof(Time)));
        si = reinterpret_cast<uint32_t *>(take((size_t)cap * 4));
        amask = reinterpret_cast<uint32_t *>(take((size_t)ns * 4));
        smask = reinterpret_cast<uint32_t *>(take((size_t)ns * WORDS * 4));
        sgroups = reinterpret_cast<uint32_t *>(take((size_t)ns * 4));
        lgroups = reinterpret_cast<uint32_t *>(take((size_t)nl * 2));
        par = reinterpret_cast<uint16_t *>(take((size_t)cap * 2));
        prev = reinterpret_cast<uint16_t *>(take((size_t)cap * 2));
        best = reinterpret_cast<uint16_t *>(take((size_t)cap * 2));
        va = reinterpret_cast<uint16_t *>(take((size_t)cap * 2));
        top = reinterpret_cast<uint16_t *>(take((size_t)cap * 2));
        jump = reinterpret_cast<uint16_t *>(take(JUMP ? (size_t)cap * 2 : 0));
        before = reinterpret_cast<uint16_t *>(take((size_t)ns * WORDS * 2));
        cbase = reinterpret_cast<uint16_t *>(take(512));
        scid = reinterpret_cast<uint16_t *>(take(512));
        dep = take(cap);
        vn = take(cap);
        sid = take(SR);
        ndep = take(256);
        slist = take(256);
        tlist = take(ns);
        last = take((size_t)WORDS * nl);
    }
    static size_t smem(int nl, int ns) {
        return (size_t)(SR + nl) * (16 + (JUMP ? 2 : 0) + 2 * sizeof(Time)) + SR + (size_t)(WORDS + 2) * nl + (size_t)ns * (8 + 6 * WORDS + 1) + 1024 + 512;
    }
};
using EncTileA = EncTile<256, 4, false, uint32_t>;
using EncTileB = EncTile<512, 2, true, uint32_t>;
using EncTileF = EncTile<256, 4, false, uint64_t>;       // the common layout for events far apart
constexpr int EN_LEVELS_A = 512, EN_STREAMS_A = 64;      // levels and streams of the common layout
constexpr int EN_LEVELS_B = 2048;                        // levels of the wide one
// Groups of streams: past the wide layout's levels, and where a step of the whole
// trace touches so many streams that carrying their open ranges on costs more than
// the partition.  300k / 4M / 20M kernels on 200 streams of 4 levels: 265 / 546 /
// 1,860 us per join by groups, 243 / 543 / 2,022 in the wide layout; on 255 streams
// 274 / 551 / 1,882 and 257 / 568 / 2,117; on 100 streams 258 / 527 / 1,817 and
// 221 / 486 / 1,795.
constexpr int EN_STREAMS_B = 160;
constexpr int64_t EN_GROUP_EVENTS = 4 << 20;
constexpr int64_t EN_TILE = 2048, EN_TILE_MIN = 512;     // events of a tile; of a part's one tile in small traces
constexpr int64_t EN_EARLY = 1 << 20;                    // events from which a join looks at the checks before the end
// Times of a step in 32 bits end it 4 s after its first event.  A block counts the
// steps that ended so.  Where the trace's span alone makes as many of them on
// average as a second run costs (a few us each: far_steps), a block with more than
// EN_FAR gives the trace up (F_TIMES_FAR), and it is taken with times in 64 bits;
// else (long gaps, a thin tail) one with four times that many does.  A join of 1M kernels
// on 8 streams with an event every 5 / 20 / 200 / 5,000 ms: 223 / 279 / 265 / 260 us,
// 221 / 331 / 1,152 / 4,516 by 32-bit steps alone; 182 with events 0.3 ms apart.
constexpr int EN_FAR = 4;
__host__ __device__ __forceinline__ int far_steps(int64_t events) { return 8 + (int)(events >> 20); }
constexpr size_t EN_SMEM_F = 74 * 1024;                  // of that layout: three blocks a multiprocessor at least, else groups

// One block per part, tile by tile; a tile with more ranges than SR, or whose
// times span 2^32 ns, is taken in steps.  A step's ranges, and the ranges open
// when it begins, lie in shared memory (times relative to the part's first
// event, or to the step's after 2^32 ns, in 32 bits; in 64 with EncTileF), and
// once per range this is worked out:
//   parent  the last range of the level above that starts no later
//   chain   Algorithm 2's result for the range and its ancestors: walking
//           outward to the first structural range, the innermost operator
//           and the number of operators
//   best    of the ranges of the stream up to this one the latest-starting
//           that has a length, the deepest of those with its start: whatever
//           contains a time after this entry's start and before the stream's
//           next one is `best` or an ancestor of it
// A kernel then takes the last range of its stream that starts by it (the
// step's ranges before the kernel are counted along the warp's kernels, the
// stream's last one among them found by its bit mask), climbs from its `best`
// past the ranges that have ended, and has its answer in the chain found
// there.  A kernel that starts with that range takes the range's own chain,
// unless another range of the stream starts or ends at that instant (D_MIXED):
// then the last range of each level up to the instant stands for its level,
// and the chain is walked along those (closed intervals).
//
// The laminar checks ride along: each range against its predecessor in its
// level, and against its parent (equal starts in array order included; where
// those go on past the loaded ranges, F_LEVEL_FIXUP asks for a run on ranges
// sorted so that parents come first).  F_LEVEL_FIXUP also reports equal starts
// of a level out of (start, end) order.  With `final` both are errors.
// Ranges that are not laminar give wrong answers but no stray access: parents
// lie one level up, so every climb and walk ends within 32 steps.
//
// Open ranges are kept from step to step, a warp to a stream and a lane to a
// level, and only for the streams that the step touched: their chains are read
// off the warp's ballots, so a range of the tile walks outward only to the
// first open one, and a step's tables are cleared by the entries it made.
//
// Bound by issue (2.4 instructions a cycle) and by the shared-memory chains of
// the links, not by HBM: 430 us for 20M kernels and 5.1M ranges on 16 streams
// of 8 levels, 1,950 us for 50M and 14.5M on 64 streams of 32 (1,990 with climbs
// of one level at a time), 14 us for 2,000.
// With every open range's chain walked, and every level's tables cleared,
// counted up and made relative to the next event at each step, 490, 3,840 and
// 17 us; steps of 1,024 ranges (one block of 1,024 threads) 2,780 us where 512
// took 2,610.  The level lists, stream partition, windows and per-stream
// tiles it replaces took 436 us in their largest kernel and another 300 us in
// eight more launches (partly side by side) for the same trace, two host waits
// and 60 us for the small one.  Also measured: one search per depth and kernel
// in level lists of the tile (1,170 us), entries grouped by stream with a
// search per kernel (696 us).
//
// GROUPS: the parts are those of groups of streams (EncGroup).
template <typename TL, bool KEYS, bool GROUPS>
__global__ void __launch_bounds__(TL::THREADS, TL::BLOCKS)
    k_enclose(EncView V, int64_t parts, int tp, const uint32_t *__restrict__ tile_r,
              const uint32_t *__restrict__ rows, const uint32_t *__restrict__ row_len, int carried,
              const uint32_t *__restrict__ lvlmask, int nlcap, int nscap, const EncGroup *__restrict__ G,
              unsigned leave_on, int final, int32_t *__restrict__ out_range,
              uint8_t *__restrict__ out_nop, DevStatus *st) {
    pdl_wait();
    constexpr int THREADS = TL::THREADS, WARPS = THREADS / 32, RPT = TL::RPT, SR = TL::SR, WORDS = TL::WORDS;
    using Time = typename TL::Time;
    constexpr Time NEVER = ~(Time)0;                 // an end past a step's times
    static_assert(THREADS >= 256, "a thread per stream");
    static_assert(WORDS == 16 && RPT * WARPS == WORDS, "half a warp per stream, 16 bits per level");
    if ((st->err & (ERR_INVALID | ERR_DEPTH)) || (st->flags & leave_on)) return;
    extern __shared__ __align__(16) unsigned char en_smem[];
    const TL S(en_smem, nlcap, nscap);
    __shared__ uint32_t wbuf[33];
    __shared__ int taken[2];
    __shared__ int ntouched;
    const int tid = threadIdx.x;
    const unsigned lane = lane_id(), warp = tid >> 5, lt = lanemask_lt();
    int64_t b = blockIdx.x;
    unsigned grp = 0;
    if (GROUPS) {
        int64_t tile0, part0;
        if (!enter_group(G, V, b, parts, tp, tile0, part0, grp)) return;
        tile_r += tile0;
        rows += part0 * LEVELS;
        row_len += part0;
    }
    // levels present: depths 0 .. ndep - 1 of each stream (a depth below a gap
    // has no parent level: its ranges are not nested)
    int nl, ns;
    {
        uint32_t n = 0;
        if (tid < 256 && (!GROUPS || tid >> GROUP_SHIFT == (int)grp)) {
            const uint32_t m = lvlmask[tid];
            n = m == 0xFFFFFFFFu ? 32u : (uint32_t)__ffs(~m) - 1u;
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<uint32_t>(n | (n ? 1u << 16 : 0u), wbuf, &tot);
        nl = (int)(tot & 0xFFFFu);
        ns = (int)(tot >> 16);
        if (nl > nlcap || ns > nscap) {
            if (b == 0 && tid == 0) set_flag(st, F_LEVELS_MANY);
            return;
        }
        if (tid < 256) {
            S.cbase[tid] = (uint16_t)(ex & 0xFFFFu);
            S.ndep[tid] = (uint8_t)n;
            S.scid[tid] = n ? (uint16_t)(ex >> 16) : (uint16_t)E_NONE;
            if (n) S.slist[ex >> 16] = (uint8_t)tid;
        }
    }
    for (int l = tid; l < (nl + 1) / 2; l += THREADS) S.lgroups[l] = 0;
    for (int i = tid; i < ns * WORDS; i += THREADS) S.smask[i] = 0;
    for (int q = tid; q < ns; q += THREADS) S.sgroups[q] = 0;
    const int64_t nt = parts * tp, events = V.K + V.R;
    int64_t r = tile_r[b * tp];
    int64_t k = tile_event(b * tp, nt, events) - r;
    __syncthreads();
    // the earliest event at or after (k, r): what has ended before it is over
    auto first_time = [&](int64_t kk, int64_t rr) {
        const long long t = kk < V.K ? V.time<KEYS>(kk) : LLONG_MAX, a = rr < V.R ? V.r_start[rr] : LLONG_MAX;
        return t < a ? t : a;
    };
    long long base = first_time(k, r), first = base;      // times are relative to base; the step's first event
    auto rel = [&](long long x) -> Time {
        const unsigned long long v = (unsigned long long)x - (unsigned long long)base;
        return x < base ? (Time)0 : (v >= (unsigned long long)NEVER - 1 ? NEVER : (Time)(v + 1));
    };
    // What a warp writes of a stream's open ranges, lane by depth: the chain of
    // each is the run of open levels above it, read off four ballots.
    auto open_ranges = [&](int q, uint32_t e0, bool live, Time a, Time z, uint32_t i) {
        const uint32_t kind = i >> 30;
        const unsigned m = __ballot_sync(0xffffffffu, live), le = lt | 1u << lane;
        const unsigned ops = __ballot_sync(0xffffffffu, live && kind == KIND_OP);
        const unsigned walls = __ballot_sync(0xffffffffu, live && kind == KIND_STRUCT);
        const unsigned longs = __ballot_sync(0xffffffffu, live && a < z);
        const unsigned gap = ~m & le;
        const unsigned lo = gap ? 32u - __clz(gap) : 0u;                         // the run's outermost level
        if (lane == 0) S.amask[q] = m;
        if (lane < WORDS) S.before[q * WORDS + lane] = m ? (uint16_t)(e0 + 31u - __clz(m)) : (uint16_t)E_NONE;
        if (!live) return;
        const uint32_t e = e0 + lane;
        const unsigned run = le & ~((1u << lo) - 1u), wall = walls & run;
        const unsigned seen = ops & (wall ? run & ~((2u << (31 - __clz(wall))) - 1u) : run);
        S.ss[e] = a;
        S.se[e] = z;
        S.si[e] = i;
        S.dep[e] = (uint8_t)(lane | D_MIXED);
        S.par[e] = lane > 0 && ((m >> (lane - 1)) & 1u) ? (uint16_t)(e - 1) : (uint16_t)E_NONE;
        S.prev[e] = m & lt ? (uint16_t)(e0 + 31u - __clz(m & lt)) : (uint16_t)E_NONE;
        S.va[e] = seen ? (uint16_t)(e0 + 31u - __clz(seen)) : (uint16_t)E_NONE;
        S.vn[e] = (uint8_t)__popc(seen);
        S.top[e] = (uint16_t)(e0 + lo);
        if (TL::JUMP) S.jump[e] = lane >= lo + 4 ? (uint16_t)(e - 4) : (uint16_t)E_NONE;
        S.best[e] = longs & le ? (uint16_t)(e0 + 31u - __clz(longs & le)) : (uint16_t)E_NONE;
    };
    for (int q = (int)warp; q < ns; q += WARPS) {                                // a warp per stream, a lane per depth
        const unsigned s = S.slist[q], l = s * 32u + lane;
        uint32_t v = 0, i = 0;
        Time a = 0, z = 0;
        if (lane < S.ndep[s]) {
            if (carried) v = rows[b * LEVELS + l];
            else
#pragma unroll 4
                for (int64_t x = 0; x < b; ++x) {
                    const uint32_t u = l < row_len[x] ? rows[x * LEVELS + l] : 0u;
                    v = u > v ? u : v;
                }
        }
        bool live = v != 0;
        if (live) {
            const long long end = V.r_end[v - 1];
            live = end >= base;
            a = rel(V.r_start[v - 1]);
            z = rel(end);
            i = (v - 1) | kind_of(V.r_op[v - 1]) << 30;
        }
        open_ranges(q, (uint32_t)SR + S.cbase[s], live, a, z, i);
    }
    bool err = false, fix = false;
    int far = 0;
    int64_t r_end_n = tile_r[b * tp + 1];           // the next step's end
    __syncthreads();
    for (int64_t t = b * tp + 1; t <= (b + 1) * tp; ++t) {
        const int64_t r1 = r_end_n, k1 = tile_event(t, nt, events) - r1;
        if (t < (b + 1) * tp) r_end_n = tile_r[t + 1];
        while (k < k1 || r < r1) {
            int nr = (int)(r1 - r < SR ? r1 - r : SR), nk = (int)(k1 - k);
            long long nbase = first_time(k + nk, r + nr);
            // ---- the step: the whole tile, or up to the first event that
            // must wait (a kernel that starts no earlier than a range not
            // loaded; 2^32 ns from base)
            auto near = [&](long long x) { return (unsigned long long)x - (unsigned long long)base < (unsigned long long)NEVER - 15; };
            const long long t_last = nk > 0 ? V.time<KEYS>(k + nk - 1) : first, a_last = nr > 0 ? V.r_start[r + nr - 1] : first;
            if (!(near(t_last) && near(a_last)) && base != first) {
                // the open ranges relative to this step's first event (once in some 4 s of the trace)
                const unsigned long long shift = (unsigned long long)first - (unsigned long long)base;
                base = first;
                for (int q = (int)warp; q < ns; q += WARPS) {
                    const unsigned s = S.slist[q];
                    const uint32_t e0 = (uint32_t)SR + S.cbase[s], e = e0 + lane;
                    Time a2 = 0, z2 = 0;
                    uint32_t i = 0;
                    if ((S.amask[q] >> lane) & 1u) {
                        const Time a = S.ss[e], z = S.se[e];
                        i = S.si[e];
                        a2 = (unsigned long long)a > shift ? a - (Time)shift : (Time)0;
                        z2 = z == NEVER ? rel(V.r_end[i & POS_MASK])
                                        : ((unsigned long long)z > shift ? z - (Time)shift : (Time)0);
                    }
                    open_ranges(q, e0, z2 > 0, a2, z2, i);
                }
                __syncthreads();
            }
            bool whole = r1 - r <= SR && near(t_last) && near(a_last);
            if (!whole) {
                if (sizeof(Time) == 4 && !(near(t_last) && near(a_last)) && ++far > EN_FAR) {
                    const uint64_t span = V.K > 0 ? (uint64_t)st->mm[MM_KSTART_MAX] - (uint64_t)st->mm[MM_KSTART_MIN] : 0;
                    const int most = far_steps(events);
                    if ((span >> 32) > (uint64_t)(most * parts) || far > 4 * most) {
                        if (tid == 0) set_flag(st, F_TIMES_FAR);
                        return;
                    }
                }
                // by two warps, 32 probes a round
                if (warp < 2) {
                    const bool more = r + nr < r1;
                    const long long next = more ? V.r_start[r + nr] : 0;
                    int lo = 0, hi = warp == 0 ? nk : nr;
                    while (lo < hi) {
                        const int step = (hi - lo + 31) >> 5, p = lo + (int)lane * step;
                        bool ok = false;
                        if (p < hi) {
                            const long long x = warp == 0 ? V.time<KEYS>(k + p) : V.r_start[r + p];
                            ok = near(x) && !(warp == 0 && more && x >= next);
                        }
                        const unsigned m = ~__ballot_sync(0xffffffffu, ok);
                        const int c = m ? __ffs(m) - 1 : 32;
                        if (c == 0) break;
                        const int nh = lo + c * step;
                        lo += (c - 1) * step + 1;
                        hi = nh < hi ? nh : hi;
                    }
                    if (lane == 0) taken[warp] = lo;
                }
                __syncthreads();
                nk = taken[0];
                nr = taken[1];
                nbase = first_time(k + nk, r + nr);
                if (nk == 0 && nr == 0) {                                // cannot happen on ordered records
                    if (tid == 0) set_err(st, ERR_INVALID);
                    return;
                }
                // kernels before every range that is taken later: with kernels
                // left over, ranges only while they start by the last one taken
                // or no kernel is (all those left start after them)
            }
            const bool more = r + nr < V.R;                              // ranges past this step's
            const long long next = more ? V.r_start[r + nr] : 0;
            // exact for the step's events
            auto rel_near = [&](long long x) { return (Time)x - (Time)base + 1u; };
            // ---- ranges, 32 at a time: the stream's and the level's earlier
            // ranges in the group by lane masks, before it by tables (links)
            uint32_t lk[RPT], pk[RPT];               // the level's range before | level << 16; parent | prev on stream << 16
            if (tid == 0) ntouched = 0;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const unsigned g = i * WARPS + warp;
                const int at = (int)g * 32, e = at + (int)lane;
                lk[i] = 0xFFFFu << 16;
                pk[i] = 0;
                if (at >= nr) continue;
                const bool in = e < nr;
                const int64_t p = r + e;
                const long long a = in ? V.r_start[p] : 0, z = in ? V.r_end[p] : 0;
                const unsigned s = in ? V.r_stream[p] : 0u, d = in ? V.r_depth[p] : 0u;
                const uint32_t op = in ? V.r_op[p] : 0u;
                const bool lvl = in && d < S.ndep[s];
                err |= in && !lvl;
                const unsigned q = lvl ? S.scid[s] : 256u;
                const unsigned ps = __match_any_sync(0xffffffffu, q);
                unsigned pl = ps, pp = ps;           // lanes of the level, of the level above
#pragma unroll
                for (int bit = 0; bit < 5; ++bit) {
                    const unsigned x = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
                    pl &= (d >> bit) & 1u ? x : ~x;
                    pp &= ((d - 1u) >> bit) & 1u ? x : ~x;
                }
                if (lvl) {
                    const unsigned c = S.cbase[s] + d;
                    const unsigned ml = pl & lt, mp = d ? pp & lt : 0u, ms = ps & lt;
                    lk[i] = (ml ? at + 32u - __clz(ml) : 0u) | c << 16;                  // index + 1, 0 not here
                    pk[i] = (mp ? at + 32u - __clz(mp) : 0u) | (ms ? at + 32u - __clz(ms) : 0u) << 16;
                    S.ss[e] = rel_near(a);
                    S.se[e] = rel(z);
                    S.si[e] = (uint32_t)p | kind_of(op) << 30;
                    S.dep[e] = (uint8_t)d;
                    S.sid[e] = (uint8_t)q;
                    if ((pl >> lane) == 1u) {                                            // the level's last of the 32
                        S.last[g * nlcap + c] = (uint8_t)lane;
                        atomicOr(&S.lgroups[c / 2], 1u << (g + 16 * (c & 1u)));
                    }
                    if (ms == 0) {
                        S.smask[q * WORDS + g] = ps;
                        atomicOr(&S.sgroups[q], 1u << g);
                    }
                } else if (in) {                     // below a gap: on no stream's chain
                    S.ss[e] = rel_near(a);
                    S.se[e] = 0;
                    S.si[e] = KIND_STRUCT << 30;
                    S.dep[e] = (uint8_t)(D_DEPTH | D_MIXED);
                    S.sid[e] = 255;
                    S.par[e] = S.prev[e] = (uint16_t)E_NONE;
                }
            }
            __syncthreads();
            // ---- links, and the laminar checks.  Relative times are exact
            // below NEVER; two clamped ends are compared as they are.
            auto last_of = [&](uint32_t l, unsigned below) -> uint32_t {                 // the level's, in groups below; + 1
                const unsigned h = (S.lgroups[l / 2] >> (16 * (l & 1u))) & ((1u << below) - 1u);
                const unsigned g = 31 - __clz(h);
                return h ? g * 32 + S.last[g * nlcap + l] + 1u : 0u;
            };
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const unsigned g = i * WARPS + warp;
                const uint32_t c = lk[i] >> 16;
                if (c == 0xFFFFu) continue;
                const uint32_t e = g * 32 + lane;
                const unsigned q = S.sid[e], d = S.dep[e] & D_DEPTH, am = S.amask[q];
                const Time a = S.ss[e];
                auto earlier = [&](uint32_t u, uint32_t l, unsigned depth) -> uint32_t {
                    if (u == 0) u = last_of(l, g);
                    return u ? u - 1 : ((am >> depth) & 1u ? (uint32_t)SR + l : (uint32_t)E_NONE);
                };
                const uint32_t y = earlier(lk[i] & 0xFFFFu, c, d);
                uint32_t p = d ? earlier(pk[i] & 0xFFFFu, c - 1, d - 1) : (uint32_t)E_NONE;
                uint32_t x = pk[i] >> 16;                                            // before it on the stream
                if (x) --x;
                else {
                    const unsigned h = S.sgroups[q] & ((1u << g) - 1u), w = 31 - __clz(h);
                    x = h ? w * 32 + 31 - __clz(S.smask[q * WORDS + w]) : (uint32_t)S.before[q * WORDS];
                }
                bool mixed = x != E_NONE && S.ss[x] == a;
                for (int f = (int)e + 1; f < nr && S.ss[f] == a; ++f) {              // equal starts further on
                    if (S.sid[f] != q) continue;
                    mixed = true;
                    if (d && (S.dep[f] & D_DEPTH) == d - 1) p = f;
                }
                auto end_of = [&](uint32_t w) { return V.r_end[S.si[w] & POS_MASK]; };
                auto ends_before = [&](uint32_t w, uint32_t v) {                     // entry w ends before entry v
                    const Time f = S.se[w], g = S.se[v];
                    return f == NEVER && g == NEVER ? end_of(w) < end_of(v) : f < g;
                };
                if (y != E_NONE) {
                    if (S.ss[y] == a && ends_before(e, y)) fix = true;               // starts with it, ends before it
                    else if (S.se[y] > a) err = true;
                    mixed |= S.se[y] == a;
                }
                if (d && (p == E_NONE || ends_before(p, e))) {
                    if (more && !final && next == V.r_start[r + e]) fix = true;
                    else err = true;
                }
                S.par[e] = (uint16_t)p;
                S.prev[e] = (uint16_t)x;
                if (mixed) S.dep[e] = (uint8_t)(d | D_MIXED);
            }
            // the last entry before each group, half a warp to a stream
            for (int q2 = (int)warp * 2; q2 < ns; q2 += WARPS * 2) {
                const int q = q2 + (int)(lane >> 4), w = (int)(lane & 15u);
                const bool some = q < ns && S.sgroups[q] != 0;
                if (!__any_sync(0xffffffffu, some)) continue;
                const uint32_t m = some ? S.smask[q * WORDS + w] : 0u;
                uint32_t u = m ? w * 32 + 32 - __clz(m) : 0u;
#pragma unroll
                for (int h = 1; h < 16; h <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xffffffffu, u, h, 16);
                    u = v > u ? v : u;
                }
                u = __shfl_up_sync(0xffffffffu, u, 1, 16);
                if (some && w > 0) S.before[q * WORDS + w] = u ? (uint16_t)(u - 1) : S.before[q * WORDS];
                if (some && w == 0) S.tlist[atomicAdd(&ntouched, 1)] = (uint8_t)q;
            }
            __syncthreads();
            // ---- the kernels: each warp an equal run, 32 at a time (the first of them on their way already)
            const int per = (nk + 32 * WARPS - 1) / (32 * WARPS) * 32;
            const int j0 = (int)warp * per, j1 = j0 + per < nk ? j0 + per : nk;
            long long t_n = 0;
            unsigned s_n = 0;
            if (j0 + (int)lane < j1) {
                t_n = V.time<KEYS>(k + j0 + lane);
                s_n = V.stream<KEYS>(k + j0 + lane);
            }
            // ---- chains and `best`, up to the first open range, which has its own
            auto best_of = [&](uint32_t e) -> uint32_t {
                while (e < SR && S.ss[e] >= S.se[e]) e = S.prev[e];                      // zero length
                if (e >= SR) return e == E_NONE ? e : (uint32_t)S.best[e];
                uint32_t w = e;
                const Time a = S.ss[e];
                for (uint32_t x = S.prev[e]; x != E_NONE && S.ss[x] == a; x = S.prev[x])
                    if (S.se[x] > a && (S.dep[x] & D_DEPTH) > (S.dep[w] & D_DEPTH)) w = x;
                return w;
            };
            for (int e = tid; e < nr; e += THREADS) {
                uint32_t ans = E_NONE, n = 0, x = e, top, far = E_NONE;
                int up = 0;
                bool on = true;
                do {
                    const uint32_t kind = S.si[x] >> 30;
                    on = on && kind != KIND_STRUCT;
                    if (on && kind == KIND_OP && n++ == 0) ans = x;
                    top = x;
                    x = S.par[x];
                    if (TL::JUMP && ++up == 4) far = x;
                } while (x < SR);
                if (x != E_NONE) {
                    if (on) {
                        if (n == 0) ans = S.va[x];
                        n += S.vn[x];
                    }
                    top = S.top[x];
                    if (TL::JUMP && up < 4) {                // on along the open ones, one slot to a level
                        far = x - (4 - up);
                        if (far < top) far = E_NONE;
                    }
                }
                if (TL::JUMP) S.jump[e] = (uint16_t)far;
                S.va[e] = (uint16_t)ans;
                S.vn[e] = (uint8_t)n;
                S.top[e] = (uint16_t)top;
                S.best[e] = (uint16_t)best_of(e);
            }
            __syncthreads();
            {
                int q0 = 0;                                                              // ranges before the run
                if (j0 < j1) {
                    const Time T0 = __shfl_sync(0xffffffffu, rel_near(t_n), 0);
                    int hi = nr;
                    while (q0 < hi) {
                        const int m = (q0 + hi) >> 1;
                        if (S.ss[m] <= T0) q0 = m + 1; else hi = m;
                    }
                }
                for (int j = j0; j < j1; j += 32) {
                    const bool in = j + (int)lane < j1;
                    const Time T = rel_near(t_n);
                    const unsigned s = s_n;
                    const int64_t kk = k + j + (int)lane;
                    if (j + 32 + (int)lane < j1) {
                        t_n = V.time<KEYS>(kk + 32);
                        s_n = V.stream<KEYS>(kk + 32);
                    }
                    // ranges that start by each kernel: those by the last one
                    // first, then each lane's share of them
                    const int top = j1 - j < 32 ? j1 - j - 1 : 31;
                    const Time Tm = __shfl_sync(0xffffffffu, T, top);
                    int qn = q0;
                    for (;;) {
                        const Time v = q0 + (int)lane < nr ? S.ss[q0 + lane] : NEVER;
                        const int c = __popc(__ballot_sync(0xffffffffu, v <= Tm));
                        int h = 0;
#pragma unroll
                        for (int i = 16; i > 0; i >>= 1) h += __shfl_sync(0xffffffffu, v, h + i - 1) <= T ? i : 0;
                        q0 += c;
                        if (c < 32) {
                            qn += h;
                            break;
                        }
                        const Time v31 = __shfl_sync(0xffffffffu, v, 31);
                        qn += h + (v31 <= T ? 1 : 0);
                    }
                    if (!in) continue;
                    uint32_t ans = E_NONE;
                    unsigned n = 0;
                    const unsigned q = S.scid[s];
                    if (q != E_NONE) {
                        // the stream's last one
                        const unsigned l = qn ? (unsigned)qn - 1u : 0u, w = q * WORDS + (l >> 5);
                        const uint32_t m = qn ? S.smask[w] & ((2u << (l & 31)) - 1u) : 0u;
                        uint32_t x = m ? (l | 31u) - __clz(m) : (uint32_t)S.before[w];
                        if (x != E_NONE) {
                            const bool at_start = S.ss[x] == T;
                            if (!at_start || !(S.dep[x] & D_MIXED)) {
                                if (!at_start) x = S.best[x];
                                if (x != E_NONE && S.se[S.top[x]] >= T) {
                                    if (TL::JUMP)
                                        for (uint32_t u = x; u != E_NONE && S.se[u] < T; u = S.jump[u]) x = u;
                                    while (S.se[x] < T) x = S.par[x];
                                    ans = S.va[x];
                                    n = S.vn[x];
                                }
                            } else {
                                // ranges that start at T stand in for the older ones of their
                                // levels, beside older ones of other levels that end at T
                                const uint32_t e = x;
                                uint32_t z = e, g = e, at = 1u << (S.dep[e] & D_DEPTH);  // deepest (last) at T; first; depths
                                for (uint32_t f = S.prev[e]; f != E_NONE && S.ss[f] == T; f = S.prev[f]) {
                                    g = f;
                                    at |= 1u << (S.dep[f] & D_DEPTH);
                                    if ((S.dep[f] & D_DEPTH) > (S.dep[z] & D_DEPTH)) z = f;
                                }
                                x = best_of(S.prev[g]);                                  // open before T
                                while (x != E_NONE && S.se[x] < T) x = S.par[x];
                                if (x == E_NONE || (S.dep[x] & D_DEPTH) <= (S.dep[z] & D_DEPTH)) x = z;
                                while (x != E_NONE) {
                                    const uint32_t kind = S.si[x] >> 30, d = S.dep[x] & D_DEPTH;
                                    if (kind == KIND_STRUCT) break;
                                    if (kind == KIND_OP && n++ == 0) ans = x;
                                    x = S.par[x];
                                    if (x != E_NONE && ((at >> (d - 1)) & 1u))           // the last of this depth at T
                                        for (x = e; (S.dep[x] & D_DEPTH) != d - 1;) x = S.prev[x];
                                }
                            }
                        }
                    }
                    const int64_t o = V.korder ? V.korder[kk] : kk;
                    int32_t range = -1;
                    if (ans != E_NONE) {
                        const uint32_t p = S.si[ans] & POS_MASK;
                        range = (int32_t)(V.perm ? V.perm[p] : p);
                    }
                    out_range[o] = range;
                    if (out_nop) out_nop[o] = (uint8_t)n;
                }
            }
            __syncthreads();
            // ---- the range each level carries on: its last one, unless it is over
            k += nk;
            r += nr;
            const unsigned long long now = (unsigned long long)nbase - (unsigned long long)base;
            const int nq = ntouched;             // the others stay (ranges that have ended are climbed past)
            for (int j = (int)warp; j < nq; j += WARPS) {
                const int q = S.tlist[j];
                const unsigned s = S.slist[q];
                const uint32_t l = S.cbase[s] + lane;
                uint32_t i = 0;
                Time a = 0, z = 0;
                bool live = false;
                if (lane < S.ndep[s]) {
                    const uint32_t u = last_of(l, WORDS), f = u ? u - 1 : (uint32_t)SR + l;
                    if (u || ((S.amask[q] >> lane) & 1u)) {
                        a = S.ss[f];
                        z = S.se[f];
                        i = S.si[f];
                        live = z == NEVER ? V.r_end[i & POS_MASK] >= nbase : (unsigned long long)z > now;
                    }
                    if (u) reinterpret_cast<uint16_t *>(S.lgroups)[l] = 0;
                }
                if (lane < WORDS) S.smask[q * WORDS + lane] = 0;
                if (lane == WORDS) S.sgroups[q] = 0;
                open_ranges(q, (uint32_t)SR + l - lane, live, a, z, i);
            }
            first = nbase;
            __syncthreads();
        }
    }
    if (final && fix) {
        err = true;
        fix = false;
    }
    if (__any_sync(0xffffffffu, fix) && lane == 0) set_flag(st, F_LEVEL_FIXUP);
    if (__any_sync(0xffffffffu, err) && lane == 0) set_err(st, ERR_NOT_NESTED);
}

// ------------------------------------------------------------------ sorted views
// Range records in the order of the sorted keys (which hold the starts), or of
// perm alone where the keys are too wide to be kept (NULL).
__global__ void k_range_gather(EncView V, const uint64_t *__restrict__ key, int shift, long long tmin,
                               const uint32_t *__restrict__ perm, int64_t *__restrict__ start,
                               int64_t *__restrict__ end, uint8_t *__restrict__ stream, uint8_t *__restrict__ depth,
                               uint32_t *__restrict__ op) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V.R; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t r = perm[i];
        start[i] = key ? tmin + (long long)(key[i] >> shift) : V.r_start[r];
        end[i] = V.r_end[r];
        stream[i] = V.r_stream[r];
        depth[i] = V.r_depth[r];
        op[i] = V.r_op[r];
    }
}

// ------------------------------------------------------------------ groups of streams
// Kernels and ranges of the view, each partitioned by one stable counting pass.
template <bool KEYS>
struct GroupDigitK {
    EncView V;
    __device__ __forceinline__ unsigned operator()(int64_t i) const { return V.stream<KEYS>(i) >> GROUP_SHIFT; }
};
template <bool KEYS>
struct GroupPlaceK {
    EncView V;
    int64_t *start;
    uint8_t *stream;
    uint32_t *order;
    __device__ __forceinline__ void operator()(int64_t i, uint32_t dest, unsigned) const {
        start[dest] = V.time<KEYS>(i);
        stream[dest] = (uint8_t)V.stream<KEYS>(i);
        order[dest] = V.korder ? V.korder[i] : (uint32_t)i;
    }
};
struct GroupDigitR {
    const uint8_t *stream;
    __device__ __forceinline__ unsigned operator()(int64_t i) const { return stream[i] >> GROUP_SHIFT; }
};
struct GroupPlaceR {
    EncView V;
    int64_t *start, *end;
    uint8_t *stream, *depth;
    uint32_t *op, *perm;
    __device__ __forceinline__ void operator()(int64_t i, uint32_t dest, unsigned) const {
        start[dest] = V.r_start[i];
        end[dest] = V.r_end[i];
        stream[dest] = V.r_stream[i];
        depth[dest] = V.r_depth[i];
        op[dest] = V.r_op[i];
        perm[dest] = V.perm ? V.perm[i] : (uint32_t)i;
    }
};
// koffs / roffs: digit-major offsets of the counting passes (kt / rt tiles each).
__global__ void k_enc_groups(const uint32_t *__restrict__ koffs, int64_t kt, int64_t K, const uint32_t *__restrict__ roffs,
                             int64_t rt, int64_t R, int64_t parts, EncGroup *__restrict__ G) {
    pdl_wait();
    __shared__ EncGroup E[N_GROUPS];
    const int g = threadIdx.x;
    auto first = [](const uint32_t *offs, int64_t tiles, int64_t n, int d) -> int64_t {
        return n == 0 ? 0 : d == N_GROUPS ? n : (int64_t)offs[d * tiles];
    };
    EncGroup &e = E[g];
    e.k0 = first(koffs, kt, K, g);
    e.r0 = first(roffs, rt, R, g);
    e.K = first(koffs, kt, K, g + 1) - e.k0;
    e.R = first(roffs, rt, R, g + 1) - e.r0;
    const int64_t n = e.K + e.R, p = n * parts / (K + R);
    e.parts = n == 0 ? 0 : (int)(p > 0 ? p : 1);
    const int64_t tp = n == 0 ? 0 : (n + e.parts * EN_TILE - 1) / (e.parts * EN_TILE);
    e.tp = (int)(tp > 0 ? tp : 1);
    __syncwarp((1u << N_GROUPS) - 1u);
    int64_t part0 = 0, tile0 = 0;
    for (int q = 0; q < g; ++q) {
        part0 += E[q].parts;
        tile0 += (int64_t)E[q].parts * E[q].tp + 1;
    }
    EncGroup out = e;
    out.part0 = (int)part0;
    out.tile0 = tile0;
    G[g] = out;
}

// ------------------------------------------------------------------ host
opattr_status enclose_verdict(const DevStatus &H, int64_t K) {
    if (H.err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
    if (H.err & ERR_DEPTH) return OPATTR_E_DEPTH;
    if (K > 0 && (H.mm[MM_KSTART_MAX] - H.mm[MM_KSTART_MIN]) >= (1ll << 55)) return OPATTR_E_INVALID_ARG;
    if (H.err & ERR_NOT_NESTED) return OPATTR_E_NOT_NESTED;
    if (H.err & ERR_TIMEOUT) return OPATTR_E_TIMEOUT;
    return OPATTR_OK;
}

// The enclosure launches on view V: the parts (already there after the
// checking pass on V itself), the carried ranges, the tiles.
struct EncBufs {
    int64_t parts;
    int tp;                      // tiles of a part
    uint32_t *tile_r, *rows, *row_len, *lvlmask;
    EncGroup *groups;            // NULL: one sequence
};
constexpr int64_t EN_DIRECT_PARTS = 32;          // up to this many: a block scans the rows before its own itself
template <typename TL, bool KEYS, bool GROUPS = false>
static void launch_tiles(Ctx &c, const EncView &V, const EncBufs &B, int nl, int ns, unsigned leave_on, bool final,
                         int32_t *out_range, uint8_t *out_nop) {
    nl = (nl + 7) & ~7;                          // (whole words in every table)
    ns = (ns + 7) & ~7;
    const size_t smem = TL::smem(nl, ns);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(k_enclose<TL, KEYS, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch(c, "enclose", k_enclose<TL, KEYS, GROUPS>, dim3((unsigned)B.parts), dim3(TL::THREADS), smem, V,
           B.parts, B.tp, (const uint32_t *)B.tile_r, (const uint32_t *)B.rows, (const uint32_t *)B.row_len,
           (int)(GROUPS || B.parts > EN_DIRECT_PARTS), (const uint32_t *)B.lvlmask, nl, ns, (const EncGroup *)B.groups,
           leave_on, (int)final, out_range, out_nop, c.d_status);
}
static void launch_carry(Ctx &c, const EncBufs &B) {
    if (B.groups || B.parts > EN_DIRECT_PARTS)
        launch(c, "enc_carry", B.groups ? k_enc_carry<true> : k_enc_carry<false>, dim3(256), dim3(1024), 0, B.rows, (const uint32_t *)B.row_len, B.parts,
               (const uint32_t *)B.lvlmask, (const EncGroup *)B.groups);
}

// Levels and streams with ranges, from the depths present on every stream.
struct LevelCount {
    int levels = 0, streams = 0;
    explicit LevelCount(const uint32_t *masks) {
        for (int s = 0; s < 256; ++s) {
            levels += masks[s] == 0xFFFFFFFFu ? 32 : __builtin_ctz(~masks[s]);
            streams += (masks[s] & 1u) != 0;
        }
    }
};

// Room for the partition by groups, and the partition: the view on it, its parts
// in B.
struct GroupArrays {
    int64_t *k_start, *r_start, *r_end;
    uint8_t *k_stream, *r_stream, *r_depth;
    uint32_t *korder, *r_op, *perm, *k_hist, *r_hist, *part, *tile_r, *row_len, *rows;
    EncGroup *groups;
    bool take(Arena &a, int64_t K, int64_t R, int64_t n_part, int64_t tiles, int64_t parts) {
        bool ok = (k_start = a.take<int64_t>(K)) && (k_stream = a.take<uint8_t>(K)) && (korder = a.take<uint32_t>(K));
        ok = ok && (k_hist = a.take<uint32_t>(radix_hist_elems(K))) && (part = a.take<uint32_t>(n_part));
        ok = ok && (r_start = a.take<int64_t>(R)) && (r_end = a.take<int64_t>(R)) && (r_stream = a.take<uint8_t>(R));
        ok = ok && (r_depth = a.take<uint8_t>(R)) && (r_op = a.take<uint32_t>(R)) && (perm = a.take<uint32_t>(R));
        ok = ok && (r_hist = a.take<uint32_t>(radix_hist_elems(R))) && (groups = a.take<EncGroup>(N_GROUPS));
        ok = ok && (tile_r = a.take<uint32_t>(tiles)) && (row_len = a.take<uint32_t>(parts));
        return ok && (rows = a.take<uint32_t>(parts * LEVELS));
    }
};
static EncView launch_groups(Ctx &c, const EncView &V, const GroupArrays &ga, EncBufs &B) {
    const uint32_t *koffs = nullptr;
    if (V.k_key) {
        koffs = digit_offsets(c, GroupDigitK<true>{V}, V.K, ga.k_hist, ga.part, N_GROUPS);
        digit_move(c, "group_kernels", GroupDigitK<true>{V}, V.K, koffs,
                   GroupPlaceK<true>{V, ga.k_start, ga.k_stream, ga.korder});
    } else {
        koffs = digit_offsets(c, GroupDigitK<false>{V}, V.K, ga.k_hist, ga.part, N_GROUPS);
        digit_move(c, "group_kernels", GroupDigitK<false>{V}, V.K, koffs,
                   GroupPlaceK<false>{V, ga.k_start, ga.k_stream, ga.korder});
    }
    const uint32_t *roffs = digit_offsets(c, GroupDigitR{V.r_stream}, V.R, ga.r_hist, ga.part, N_GROUPS);
    digit_move(c, "group_ranges", GroupDigitR{V.r_stream}, V.R, roffs,
               GroupPlaceR{V, ga.r_start, ga.r_end, ga.r_stream, ga.r_depth, ga.r_op, ga.perm});
    auto tiles = [](int64_t n) { return (n + RADIX_TILE - 1) / RADIX_TILE; };
    launch(c, "enc_groups", k_enc_groups, dim3(1), dim3(N_GROUPS), 0, koffs, tiles(V.K), V.K, roffs, tiles(V.R), V.R,
           B.parts, ga.groups);
    EncView G{};
    G.k_start = ga.k_start;
    G.k_stream = ga.k_stream;
    G.korder = ga.korder;
    G.K = V.K;
    G.r_start = ga.r_start;
    G.r_end = ga.r_end;
    G.r_stream = ga.r_stream;
    G.r_depth = ga.r_depth;
    G.r_op = ga.r_op;
    G.perm = ga.perm;
    G.R = V.R;
    B.parts += N_GROUPS;             // rounded up to one part at least for every group
    B.tile_r = ga.tile_r;
    B.row_len = ga.row_len;
    B.rows = ga.rows;
    B.groups = ga.groups;
    return G;
}

opattr_status do_enclose(Ctx &c, const opattr_kernels *kern, const opattr_ranges *rng, int32_t *out_range,
                         uint8_t *out_nop) {
    const int64_t K = kern->n, R = rng->n;
    if (K < 0 || R < 0 || R >= (1ll << 30) || K >= (1ll << 31)) return OPATTR_E_INVALID_ARG;
    if (K > 0 && (!kern->stream || !kern->start_ns || !out_range)) return OPATTR_E_INVALID_ARG;
    if (R > 0 && (!rng->stream || !rng->start_ns || !rng->end_ns || !rng->depth || !rng->op_id))
        return OPATTR_E_INVALID_ARG;

    EncBufs B{};
    B.parts = std::max<int64_t>(1, std::min<int64_t>((K + R + EN_TILE_MIN - 1) / EN_TILE_MIN,
                                                     (int64_t)sm_count(c) * EncTileA::BLOCKS));
    B.tp = (int)std::max<int64_t>(1, (K + R + B.parts * EN_TILE - 1) / (B.parts * EN_TILE));
    const int64_t tiles = B.parts * B.tp;
    Need nd;
    nd.add<uint32_t>(tiles + 1).add<uint32_t>(B.parts).add<uint32_t>(B.parts * LEVELS).add<uint32_t>(256);
    if (c.agg_words > 0) nd.add<uint32_t>(c.agg_words);
    const bool keep_order = c.in_join && K > 0;       // a join keeps the time order for its matching
    if (keep_order) nd.add<uint32_t>(K);
    opattr_status st = ensure_arena(c, std::max(nd.bytes + 4096, c.join_scratch));
    if (st) return st;
    Arena a(c);
    // first, at the start of the arena, what outlives the enclosure
    uint32_t *agg = c.agg_words > 0 ? a.take<uint32_t>(c.agg_words) : nullptr;
    uint32_t *kept_order = keep_order ? a.take<uint32_t>(K) : nullptr;
    B.lvlmask = a.take<uint32_t>(256);
    B.tile_r = a.take<uint32_t>(tiles + 1);
    B.row_len = a.take<uint32_t>(B.parts);
    B.rows = a.take<uint32_t>(B.parts * LEVELS);
    if (!B.lvlmask || !B.tile_r || !B.row_len || !B.rows) return OPATTR_E_OOM;
    const ZeroRun z[2] = {{B.lvlmask, 256}, {agg, agg ? c.agg_words : 0}};
    if ((st = reset_status(c, 2, z))) return st;

    EncView V{};
    V.k_start = kern->start_ns;
    V.k_stream = kern->stream;
    V.K = K;
    V.r_start = rng->start_ns;
    V.r_end = rng->end_ns;
    V.r_stream = rng->stream;
    V.r_depth = rng->depth;
    V.r_op = rng->op_id;
    V.R = R;
    auto al = [](const void *p, uintptr_t n) { return (reinterpret_cast<uintptr_t>(p) & (n - 1)) == 0; };
    EncCheck C{};
    C.vec = al(kern->start_ns, 16) && al(kern->stream, 8);
    c.spec_ran = c.spec_k > 0;
    if (c.spec_ran) {
        C.kname = c.spec_kname;
        C.nname = c.spec_nname;
        C.idx = c.spec_idx;
        C.kind = c.spec_kind;
        C.pair_vec = al(C.kname, 16) && al(C.nname, 16) && al(C.idx, 16) && al(C.kind, 8);
    }
    c.max_known = c.max_ncu != nullptr;
    if (c.max_ncu) {
        C.mk = kern->name_id;
        C.mn = c.max_ncu->name_id;
        C.ms = c.max_ncu->stream;
        C.M = c.max_ncu->n;
    }
    launch(c, "enc_parts", k_enc_parts<true, false>, dim3((unsigned)B.parts), dim3(EP_THREADS), 0, V, C, B.parts,
           B.tp, B.tile_r, B.rows, B.row_len, B.lvlmask, (const EncGroup *)nullptr, c.d_status);
    // a large join looks at the checks' verdict while the rest runs on the
    // taking that the records are in order; a small one reads it once, at its end
    const bool early = c.defer_status && K + R >= EN_EARLY;
    const SmallCopy masks{c.h_small, B.lvlmask, 256 * sizeof(uint32_t)};
    if (early && (st = post_status(c, 1, &masks))) return st;
    launch_carry(c, B);
    // (the run of a join that is redone would leave as it did before, but for wider times)
    const unsigned again = c.redo & ~F_LEVEL_FIXUP;
    const bool run = again == 0 || again == F_TIMES_FAR;
    if (run)
        (again ? launch_tiles<EncTileF, false> : launch_tiles<EncTileA, false>)(
            c, V, B, EN_LEVELS_A, EN_STREAMS_A, F_K_UNSORTED | F_R_UNSORTED, false, out_range, out_nop);
    if (c.defer_status) {
        bool usual = true;
        if (early) {
            if ((st = await_status(c))) return st;
            const LevelCount n(c.h_small);
            usual = !(c.h_status->flags & (F_K_UNSORTED | F_R_UNSORTED)) && n.levels <= EN_LEVELS_A &&
                    n.streams <= EN_STREAMS_A;
        }
        if (usual) {
            // the rest of the verdict comes with the aggregation's status, which the join checks
            c.enclose_k_sorted = 1;
            c.enclose_pending = true;
            return OPATTR_OK;
        }
    }
    if ((st = read_status(c, 1, &masks))) return st;
    bool k_sorted = !(c.h_status->flags & F_K_UNSORTED), r_sorted = !(c.h_status->flags & F_R_UNSORTED);
    c.enclose_k_sorted = k_sorted ? 1 : 0;
    const LevelCount present(c.h_small);
    const bool many = present.levels > EN_LEVELS_A || present.streams > EN_STREAMS_A;
    // (with a span of so many steps the 32-bit times need no try; nor in the wide
    // layout, which is no faster than wider times in the common one, with a step of
    // 4 s for every four tiles)
    const uint64_t span = K > 0 ? (uint64_t)c.h_status->mm[MM_KSTART_MAX] - (uint64_t)c.h_status->mm[MM_KSTART_MIN] : 0;
    const bool far_fits = !many || EncTileF::smem(present.levels + 7, present.streams + 7) <= EN_SMEM_F;
    const bool gave_up = (c.h_status->flags & F_TIMES_FAR) != 0;
    bool far = gave_up || (c.redo & F_TIMES_FAR) || (span >> 32) > (uint64_t)(far_steps(K + R) * B.parts) ||
               (many && far_fits && (span >> 30) > (uint64_t)tiles);
    const bool grouped = present.levels > EN_LEVELS_B || (present.streams > EN_STREAMS_B && K + R > EN_GROUP_EVENTS) ||
                         (far && !far_fits);
    const bool fixup = (c.h_status->flags & F_LEVEL_FIXUP) != 0;
    if ((st = enclose_verdict(*c.h_status, K)) && !((fixup || gave_up) && st == OPATTR_E_NOT_NESTED)) return st;
    if (run && k_sorted && r_sorted && !many && !fixup && !gave_up) return OPATTR_OK;

    // ---- records out of order, ranges of one level that share a start and are
    // out of (start, end) order, more levels than the common layout holds, or
    // events far apart: the tiles again, on the sorted view, with room for every
    // level or by groups, with wider times
    const unsigned names_differ = c.h_status->flags & F_NAMES_DIFFER;   // the pairing's verdict stays
    const long long rmin = c.h_status->mm[MM_RSTART_MIN], rmax = c.h_status->mm[MM_REND_MAX];
    const long long kmin = c.h_status->mm[MM_KSTART_MIN];
    int nks = 0;                                  // streams with kernels
    uint8_t *scmap = c.h_stage, *unmap = c.h_stage + 256;
    memset(c.h_stage, 0, 512);
    for (int s = 0; s < 256; ++s)
        if ((c.h_status->kstreams[s >> 5] >> (s & 31)) & 1u) {
            scmap[s] = (uint8_t)nks;
            unmap[nks++] = (uint8_t)s;
        }
    size_t more = 0;
    if (!k_sorted) more += time_sort_scratch(K) + 512 + 4096;
    {
        Need n2;
        n2.add<int64_t>(R).add<int64_t>(R).add<uint8_t>(R).add<uint8_t>(R).add<uint32_t>(R);
        more += n2.bytes + time_sort_scratch(R) + 4096;
    }
    const int64_t g_parts = B.parts + N_GROUPS, g_tiles = (K + R) / EN_TILE + B.parts + 3 * N_GROUPS;
    const int64_t g_part = scan_scratch_elems(std::max(radix_hist_elems(K), radix_hist_elems(R)));
    if (grouped) {
        Need n3;
        n3.add<int64_t>(K).add<uint8_t>(K).add<uint32_t>(K).add<uint32_t>(radix_hist_elems(K)).add<uint32_t>(g_part);
        n3.add<int64_t>(R).add<int64_t>(R).add<uint8_t>(R).add<uint8_t>(R).add<uint32_t>(R).add<uint32_t>(R);
        n3.add<uint32_t>(radix_hist_elems(R)).add<EncGroup>(N_GROUPS).add<uint32_t>(g_tiles).add<uint32_t>(g_parts);
        more += n3.add<uint32_t>(g_parts * LEVELS).bytes + 4096;
    }
    // growing the arena keeps the prefix taken so far
    c.arena_keep = (c.arena_used + 255) & ~(size_t)255;
    {
        const char *before = c.arena;
        st = ensure_arena(c, more);
        c.arena_keep = 0;
        if (st) return st;
        const ptrdiff_t moved = c.arena - before;
        auto shift = [&](uint32_t *&p) { if (p) p = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(p) + moved); };
        shift(kept_order);
        shift(B.lvlmask);
        shift(B.tile_r);
        shift(B.row_len);
        shift(B.rows);
    }
    if (!k_sorted && K > 0) {
        unsigned char *d_map = a.take<unsigned char>(512);
        if (!d_map) return OPATTR_E_OOM;
        if ((st = copy_small(c, d_map, c.h_stage, 512, cudaMemcpyHostToDevice))) return st;
        // keyed by the compact ids of the streams with kernels
        const int sbits = bits_for((uint64_t)(nks - 1));
        uint64_t *keys = nullptr;
        uint32_t *korder = nullptr;
        if ((st = kernel_time_order(c, a, kern->stream, kern->start_ns, K, &korder, d_map, sbits, &keys))) return st;
        V.k_key = keys;
        V.k_tmin = kmin;
        V.k_sbits = sbits;
        V.k_unmap = d_map + 256;
        V.korder = korder;
        if (kept_order) {
            cudaMemcpyAsync(kept_order, korder, sizeof(uint32_t) * K, cudaMemcpyDeviceToDevice, c.stream);
            c.join_korder = kept_order;
            c.arena_keep = (size_t)(reinterpret_cast<char *>(kept_order + K) - c.arena + 255) & ~(size_t)255;
        }
    }
    const EncView raw = V;
    int64_t *gs = a.take<int64_t>(R), *ge = a.take<int64_t>(R);
    uint8_t *gt = a.take<uint8_t>(R), *gd = a.take<uint8_t>(R);
    uint32_t *go = a.take<uint32_t>(R);
    if (!gs || !ge || !gt || !gd || !go) return OPATTR_E_OOM;
    // ranges sorted so that parents come first: their verdict is final
    bool sort_ranges = !r_sorted || fixup, sorted = false;
    bool have_parts = k_sorted && !sort_ranges && !grouped;       // (too many levels only: the checking pass's parts stand)
    GroupArrays ga{};
    if (grouped && !ga.take(a, K, R, g_part, g_tiles, g_parts)) return OPATTR_E_OOM;
    for (int attempt = 0; attempt < 3; ++attempt) {
        if (sort_ranges && R > 0) {
            uint64_t *ko = nullptr;
            uint32_t *perm = nullptr;
            if ((st = range_time_order(c, a, rng->start_ns, rng->end_ns, rng->depth, R, rmin, rmax, &perm, &ko)))
                return st;
            launch(c, "range_gather", k_range_gather, dim3(grid_for(R, 256, 65535)), dim3(256), 0, raw,
                   (const uint64_t *)ko, RANGE_KEY_SHIFT, rmin, (const uint32_t *)perm, gs, ge, gt, gd, go);
            V.r_start = gs;
            V.r_end = ge;
            V.r_stream = gt;
            V.r_depth = gd;
            V.r_op = go;
            V.perm = perm;
            sort_ranges = false;
            sorted = true;
        }
        const ZeroRun zs{c.d_status, 2};              // err and flags
        if ((st = zero_runs(c, 1, &zs))) return st;
        const bool keys = V.k_key != nullptr;
        if (grouped) {
            EncBufs BG = B;
            const EncView VG = launch_groups(c, V, ga, BG);
            launch(c, "enc_view", k_enc_parts<false, false, true>, dim3((unsigned)BG.parts), dim3(EP_THREADS), 0, VG,
                   EncCheck{}, BG.parts, BG.tp, BG.tile_r, BG.rows, BG.row_len, BG.lvlmask, (const EncGroup *)BG.groups,
                   c.d_status);
            launch_carry(c, BG);
            (far ? launch_tiles<EncTileF, false, true> : launch_tiles<EncTileA, false, true>)(
                c, VG, BG, EN_LEVELS_A, EN_STREAMS_A, 0u, sorted, out_range, out_nop);
        } else if (!have_parts) {
            launch(c, "enc_view", keys ? k_enc_parts<false, true> : k_enc_parts<false, false>, dim3((unsigned)B.parts),
                   dim3(EP_THREADS), 0, V, EncCheck{}, B.parts, B.tp, B.tile_r, B.rows, B.row_len, B.lvlmask,
                   (const EncGroup *)nullptr, c.d_status);
            launch_carry(c, B);
            have_parts = true;
        }
        if (!grouped && far)
            (keys ? launch_tiles<EncTileF, true> : launch_tiles<EncTileF, false>)(
                c, V, B, std::max(EN_LEVELS_A, present.levels), std::max(EN_STREAMS_A, present.streams), 0u, sorted, out_range,
                out_nop);
        else if (!grouped && !many)
            (keys ? launch_tiles<EncTileA, true> : launch_tiles<EncTileA, false>)(c, V, B, EN_LEVELS_A, EN_STREAMS_A, 0u, sorted,
                                                                                  out_range, out_nop);
        else if (!grouped)
            (keys ? launch_tiles<EncTileB, true> : launch_tiles<EncTileB, false>)(c, V, B, present.levels, present.streams, 0u,
                                                                                  sorted, out_range, out_nop);
        if ((st = read_status(c))) return st;
        if (c.h_status->flags & F_TIMES_FAR) {
            far = true;
            continue;
        }
        if ((c.h_status->flags & F_LEVEL_FIXUP) && !sorted) {
            sort_ranges = true;
            have_parts = false;
            continue;
        }
        c.h_status->flags |= names_differ;
        return enclose_verdict(*c.h_status, K);
    }
    return OPATTR_E_CUDA;
}

}  // namespace opattr
