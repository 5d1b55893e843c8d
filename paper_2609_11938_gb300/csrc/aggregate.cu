// aggregate.cu -- per-operator aggregation, Eq. (1) and Sec. 3.8.1, with the
// rule of each counter from Table 8, and the attributed / unattributed
// totals of Fig. 4.
//
// Operators are keyed by op id (op_id[range_of_kernel[k]]), so ranges that
// share an op id aggregate together and no order of kernels or ranges is
// needed.  Three passes over the kernels and one over the ops:
//   count  validate each kernel, add up the totals, count kernels per op id
//          and give each kernel its slot among its op's kernels
//   scan   per-op offsets into one list of attributed kernels
//   place  put each attributed kernel in its slot of its op's segment
//   ops    one thread per op id accumulates its segment in ascending kernel
//          index -- the order the count's atomics left is not used, so
//          results do not depend on it -- and writes the op's record; ops
//          without kernels get empty records in the same pass.
// Accumulation is float-float with exact int64 weights (ff.cuh).
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "ff.cuh"
#include "sort.cuh"
#include "util.cuh"

namespace opattr {

constexpr int NC = OPATTR_N_COUNTERS;
// Table 8, counter #k at index k-1: SUM #1 #2 #3 #11 #15 #19, MAX #18 #20,
// duration-weighted mean for the other twelve.
constexpr int N_SUM = 6, N_DW = 12, N_MAX = 2;

struct AggIn {
    const int64_t *dur;
    const int32_t *ncu_idx;
    const float *counters;
    int64_t M;                  // ncu rows: a row index at or past M is never read (the count pass reports it)
    int64_t n_ops;
    uint32_t lane_max;          // longest op that one lane takes
    int chunk;                  // op ids of a chunk of the ops pass
    unsigned *ctr;              // [0] chunks drawn in the ops pass, [1] ops listed in dirty, [2] in mids, [3] in longs,
                                // [4] blocks done (here), [5] nonident, [6] blocks done (count); zeroed before it
    uint32_t *dirty;            // ops whose fast sums saw a null or infinite value
    uint32_t *mids;             // ops longer than a lane takes: a block each (k_agg_mid)
    uint32_t *longs;            // ops longer than a block takes: the pieces pass
    const unsigned *nonident;   // nonzero unless ncu_idx[k] == k for every kernel (set by the count pass)
    opattr_op_aggregates out;
};

// One operator's running aggregate.
//  kc, dsum       attributed kernels and their summed duration
//  mc, dall       matched kernels (with a row) and their summed duration
//  s[i]           SUM counters, float-float
//  w[i], nanw[i]  DW counters: sum of m*d, float-float, and the duration of
//                 matched kernels whose value was null (weight = dall - nanw)
//  mx[i]          MAX counters
constexpr int RENORM = 128;

// Per-counter finishing steps, kept out of line: they run once per operator
// and counter, and one copy keeps the kernel's instruction footprint small.
__device__ __noinline__ double finish_sum(float hi, float lo) {
    ff v{hi, lo};
    ff_renorm(v);
    return ff_to_f64_fast(v);
}
__device__ __noinline__ double finish_dw(float hi, float lo, long long den) {
    ff v{hi, lo};
    ff_renorm(v);
    return ff_div_to_f64(v, split_i64(den));
}
__device__ __noinline__ double finish_max(float x) { return f32_to_f64_fast(x); }
constexpr unsigned ALL_COUNTERS = (1u << NC) - 1;

// A duration as a normalised pair (as split_i64), the common case (< 2^48 ns)
// without branches.
__device__ __forceinline__ ff split_dur(long long d) {
    const unsigned long long u = (unsigned long long)d;
    if (u >> 48) return split_i64(d);
    const float a = __uint2float_rn((unsigned)(u >> 24)) * 16777216.0f;   // exact
    const float b = __uint2float_rn((unsigned)(u & 0xFFFFFFu));            // exact
    return fast_two_sum(a, b);                                            // |a| >= |b| or a == 0
}

struct Acc {
    int kc, mc;
    long long dsum, dall;
    ff s[N_SUM];
    ff w[N_DW];
    long long nanw[N_DW];
    float mx[N_MAX];
    unsigned seen;      // bit c: counter c had a non-null value
    int bad;            // an infinite counter was seen
    int terms;          // accumulations since the last renormalisation

    __device__ __forceinline__ void init() {
        kc = mc = 0;
        dsum = dall = 0;
#pragma unroll
        for (int i = 0; i < N_SUM; ++i) s[i] = ff{0.f, 0.f};
#pragma unroll
        for (int i = 0; i < N_DW; ++i) { w[i] = ff{0.f, 0.f}; nanw[i] = 0; }
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) mx[i] = -INFINITY;
        seen = 0;
        bad = 0;
        terms = 0;
    }

    __device__ __forceinline__ static int sum_col(int i) {
        return i == 0 ? 0 : i == 1 ? 1 : i == 2 ? 2 : i == 3 ? 10 : i == 4 ? 14 : 18;
    }
    __device__ __forceinline__ static int dw_col(int i) { return i < 7 ? 3 + i : (i < 10 ? 4 + i : 5 + i); }
    __device__ __forceinline__ static int max_col(int i) { return i == 0 ? 17 : 19; }

    // Adds one kernel: duration d, and its counter row when `matched`.
    __device__ __forceinline__ void accumulate(long long d, bool matched, const float4 *row) {
        kc++;
        dsum += d;
        if (!matched) return;
        mc++;
        dall += d;
        float v[NC];
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) {
            const float4 x = row[q];
            v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
        }
        float z = 0.f;              // NaN iff some value is NaN or infinite
#pragma unroll
        for (int c = 0; c < NC; ++c) z = __fmaf_rn(v[c], 0.f, z);
        unsigned valid = ALL_COUNTERS;
        if (z != z) {
            // rare: null (NaN) values take no part -- a zero value with a
            // zero weight for the sums, -inf for the maxima -- and their
            // durations leave the DW weights; infinite values are errors
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                if (isnan(v[c])) {
                    valid &= ~(1u << c);
                    v[c] = (c == 17 || c == 19) ? -INFINITY : 0.f;
                } else if (isinf(v[c])) {
                    bad = 1;
                    valid &= ~(1u << c);
                    v[c] = (c == 17 || c == 19) ? -INFINITY : 0.f;
                }
            }
#pragma unroll
            for (int i = 0; i < N_DW; ++i)
                if (!((valid >> dw_col(i)) & 1u)) nanw[i] += d;
        }
        seen |= valid;
        const ff dd = split_i64(d);
#pragma unroll
        for (int i = 0; i < N_SUM; ++i) ff_accum(s[i], v[sum_col(i)], 0.f);
#pragma unroll
        for (int i = 0; i < N_DW; ++i) {
            const ff p = mul_split(v[dw_col(i)], dd);
            ff_accum(w[i], p.hi, p.lo);
        }
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) mx[i] = fmaxf(mx[i], v[max_col(i)]);
        if (++terms >= RENORM) {
            terms = 0;
#pragma unroll
            for (int i = 0; i < N_SUM; ++i) ff_renorm(s[i]);
#pragma unroll
            for (int i = 0; i < N_DW; ++i) ff_renorm(w[i]);
        }
    }

    __device__ __forceinline__ void write(const AggIn &A, int64_t op) const {
        A.out.kernel_count[op] = kc;
        A.out.total_duration_ns[op] = dsum;
        A.out.matched_count[op] = mc;
        double *agg = A.out.agg;
        const int64_t n = A.n_ops;
        const double qnan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
        for (int i = 0; i < N_SUM; ++i)
            agg[(int64_t)sum_col(i) * n + op] = ((seen >> sum_col(i)) & 1u) ? finish_sum(s[i].hi, s[i].lo) : qnan;
#pragma unroll
        for (int i = 0; i < N_DW; ++i) {
            const long long den = dall - nanw[i];
            agg[(int64_t)dw_col(i) * n + op] =
                (((seen >> dw_col(i)) & 1u) && den > 0) ? finish_dw(w[i].hi, w[i].lo, den) : qnan;
        }
#pragma unroll
        for (int i = 0; i < N_MAX; ++i)
            agg[(int64_t)max_col(i) * n + op] = ((seen >> max_col(i)) & 1u) ? finish_max(mx[i]) : qnan;
    }

    // Row fetched from global memory (general path).
    __device__ __forceinline__ void add(const AggIn &A, int64_t k) {
        const long long d = A.dur[k];
        const int32_t j = A.ncu_idx[k];
        const bool ok = j >= 0 && j < A.M;
        accumulate(d, ok, reinterpret_cast<const float4 *>(A.counters + (int64_t)(ok ? j : 0) * NC));
    }
};

// The common case, without per-value tests: a null (NaN) or infinite value
// anywhere poisons a sum, and the op is then done again with Acc, which
// handles nulls and flags infinities.  Every counter of every matched kernel is
// non-null here, so a counter is defined iff some kernel matched, and the DW
// weight is dall.
//
// Counters go two to a register through the packed fp32 instructions (97M warp
// instructions for 4M kernels against 152M), neighbours as they lie in the row:
// a pair of DW counters weighs the duration, SUM beside DW weighs (1, duration)
// -- exact, 1 * x + 0 -- and the two MAX counters ride along as probes (their sums are not used; should one overflow, the op is done
// again like any with an infinite value).
struct AccF {
    static constexpr int PAIRS = NC / 2;
    int mc;
    long long dsum, dall;
    f32x2 hi[PAIRS], lo[PAIRS];     // counters 2p, 2p + 1: float-float sums
    float mx[N_MAX];
    int terms;

    __device__ __forceinline__ void init() {
        mc = 0;
        dsum = dall = 0;
#pragma unroll
        for (int p = 0; p < PAIRS; ++p) hi[p] = lo[p] = 0ull;
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) mx[i] = -INFINITY;
        terms = 0;
    }

    __device__ __forceinline__ void accumulate(long long d, bool matched, const float4 *row) {
        dsum += d;
        if (!matched) return;
        mc++;
        dall += d;
        f32x2 v[PAIRS];
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) {
            const ulonglong2 x = reinterpret_cast<const ulonglong2 *>(row)[q];
            v[2 * q] = x.x;
            v[2 * q + 1] = x.y;
        }
        add(d, v);
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) mx[i] = fmaxf(mx[i], f2_unpack(v[Acc::max_col(i) / 2]).y);
    }

    // One row's values into the sums.
    __device__ __forceinline__ void add(long long d, const f32x2 (&v)[PAIRS]) {
        const ff dd = split_dur(d);
        const f32x2 dw = f2_pack(dd.hi, dd.hi), dn = f2_pack(-dd.hi, -dd.hi), dl = f2_pack(dd.lo, dd.lo);
        const f32x2 sw = f2_pack(1.f, dd.hi), sn = f2_pack(-1.f, -dd.hi), sl = f2_pack(0.f, dd.lo);
#pragma unroll
        for (int p = 0; p < PAIRS; ++p) {
            if (p == 0 || p == 9) f2_accum(hi[p], lo[p], v[p]);                                     // SUM SUM, SUM MAX
            else if (p == 1 || p == 5 || p == 7) f2_accum_mul(hi[p], lo[p], v[p], sw, sn, sl);      // SUM DW
            else f2_accum_mul(hi[p], lo[p], v[p], dw, dn, dl);                                      // DW DW, DW MAX
        }
        if (++terms >= RENORM) {
            terms = 0;
#pragma unroll
            for (int p = 0; p < PAIRS; ++p) f2_renorm(hi[p], lo[p]);
        }
    }

    // counter c's sum
    __device__ __forceinline__ ff sum(int c) const {
        const float2 h = f2_unpack(hi[c / 2]), l = f2_unpack(lo[c / 2]);
        return c & 1 ? ff{h.y, l.y} : ff{h.x, l.x};
    }

    // True when no null or infinite value took part (then write() is exact to spec).
    __device__ __forceinline__ bool clean() const {
        f32x2 z = 0ull;
#pragma unroll
        for (int p = 0; p < PAIRS; ++p) z = f2_fma(f2_add(hi[p], lo[p]), 0ull, z);
        const float2 r = f2_unpack(z);
        return __fadd_rn(r.x, r.y) == 0.f;
    }

    __device__ __forceinline__ void write(const AggIn &A, int64_t op, int kc) const {
        A.out.kernel_count[op] = kc;
        A.out.total_duration_ns[op] = dsum;
        A.out.matched_count[op] = mc;
        double *agg = A.out.agg;
        const int64_t n = A.n_ops;
        const double qnan = __longlong_as_double(0x7FF8000000000000ll);
        if (mc == 0) {
            // no matched kernel: every counter is null; nothing to convert
#pragma unroll
            for (int c = 0; c < NC; ++c) agg[(int64_t)c * n + op] = qnan;
            return;
        }
#pragma unroll
        for (int i = 0; i < N_SUM; ++i) {
            ff x = sum(Acc::sum_col(i));
            ff_renorm(x);
            agg[(int64_t)Acc::sum_col(i) * n + op] = ff_to_f64_fast(x);
        }
        if (dall > 0) {
            const ff rcp = ff_recip_i64(dall);
#pragma unroll
            for (int i = 0; i < N_DW; ++i)
                agg[(int64_t)Acc::dw_col(i) * n + op] = ff_mul_to_f64(sum(Acc::dw_col(i)), rcp);
        } else {
#pragma unroll
            for (int i = 0; i < N_DW; ++i) agg[(int64_t)Acc::dw_col(i) * n + op] = qnan;
        }
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) agg[(int64_t)Acc::max_col(i) * n + op] = f32_to_f64_fast(mx[i]);
    }
};

// AccF with nulls left out and infinite values reported, as Acc has it: a value
// that takes no part adds zero, and its kernel's duration leaves that DW
// counter's weight.
struct AccN {
    AccF f;
    long long nanw[N_DW];
    unsigned seen;
    int bad;

    __device__ __forceinline__ void init() {
        f.init();
#pragma unroll
        for (int i = 0; i < N_DW; ++i) nanw[i] = 0;
        seen = 0;
        bad = 0;
    }

    __device__ __forceinline__ void accumulate(long long d, bool matched, const float4 *row) {
        f.dsum += d;
        if (!matched) return;
        f.mc++;
        f.dall += d;
        f32x2 v[AccF::PAIRS], z = 0ull;
#pragma unroll
        for (int q = 0; q < NC / 4; ++q) {
            const ulonglong2 x = reinterpret_cast<const ulonglong2 *>(row)[q];
            v[2 * q] = x.x;
            v[2 * q + 1] = x.y;
        }
        // (fmaxf passes a null over; an infinite one fails the call)
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) f.mx[i] = fmaxf(f.mx[i], f2_unpack(v[Acc::max_col(i) / 2]).y);
#pragma unroll
        for (int p = 0; p < AccF::PAIRS; ++p) z = f2_fma(v[p], 0ull, z);
        const float2 zz = f2_unpack(z);
        unsigned valid = ALL_COUNTERS;
        if (__fadd_rn(zz.x, zz.y) != 0.f) {          // NaN iff some value is NaN or infinite
            unsigned inf = 0;
#pragma unroll
            for (int p = 0; p < AccF::PAIRS; ++p) {
                float2 x = f2_unpack(v[p]);
                const unsigned a = __float_as_uint(x.x) & 0x7FFFFFFFu, b = __float_as_uint(x.y) & 0x7FFFFFFFu;
                if (a >= 0x7F800000u) {
                    valid &= ~(1u << (2 * p));
                    inf |= a == 0x7F800000u;
                    x.x = 0.f;
                }
                if (b >= 0x7F800000u) {
                    valid &= ~(2u << (2 * p));
                    inf |= b == 0x7F800000u;
                    x.y = 0.f;
                }
                v[p] = f2_pack(x.x, x.y);
            }
            bad |= (int)inf;
#pragma unroll
            for (int i = 0; i < N_DW; ++i)
                if (!((valid >> Acc::dw_col(i)) & 1u)) nanw[i] += d;
        }
        seen |= valid;
        f.add(d, v);
    }

    __device__ __forceinline__ void write(const AggIn &A, int64_t op, int kc) const {
        A.out.kernel_count[op] = kc;
        A.out.total_duration_ns[op] = f.dsum;
        A.out.matched_count[op] = f.mc;
        double *agg = A.out.agg;
        const int64_t n = A.n_ops;
        const double qnan = __longlong_as_double(0x7FF8000000000000ll);
#pragma unroll
        for (int i = 0; i < N_SUM; ++i) {
            const int c = Acc::sum_col(i);
            ff x = f.sum(c);
            ff_renorm(x);
            agg[(int64_t)c * n + op] = ((seen >> c) & 1u) ? ff_to_f64_fast(x) : qnan;
        }
#pragma unroll
        for (int i = 0; i < N_DW; ++i) {
            const int c = Acc::dw_col(i);
            const long long den = f.dall - nanw[i];
            ff x = f.sum(c);
            ff_renorm(x);
            agg[(int64_t)c * n + op] = (((seen >> c) & 1u) && den > 0) ? ff_div_to_f64(x, split_dur(den)) : qnan;
        }
#pragma unroll
        for (int i = 0; i < N_MAX; ++i) {
            const int c = Acc::max_col(i);
            agg[(int64_t)c * n + op] = ((seen >> c) & 1u) ? f32_to_f64_fast(f.mx[i]) : qnan;
        }
    }
};

// The range of kernel k; without range_of_kernel, r_op holds one operator
// per kernel and the kernel is its own "range" when it has one.
__device__ __forceinline__ int32_t range_of(const int32_t *rok, const uint32_t *r_op, int64_t k) {
    return rok ? rok[k] : (r_op[k] != OPATTR_OP_NONE ? (int32_t)k : -1);
}
template <bool DIRECT>           // DIRECT: one operator per kernel (no range_of_kernel)
__device__ __forceinline__ int32_t range_of_t(const int32_t *rok, const uint32_t *r_op, int64_t k) {
    if (DIRECT) return r_op[k] != OPATTR_OP_NONE ? (int32_t)k : -1;
    return rok[k];
}

// Within a join whose enclosure's verdict is still to be read (pending): the
// enclosure found records out of order, more levels than its layout holds, events
// too far apart or an error, and did not write all there is to aggregate.
__device__ __forceinline__ bool stopped(const DevStatus *st) {
    return (st->err & (ERR_INVALID | ERR_DEPTH)) || (st->flags & (F_REDO & ~F_LEVEL_FIXUP));
}

// ------------------------------------------------------------------ count
// Per kernel: duration >= 0, range index in [-1, R), an attributed range is
// an operator below n_ops, row index in [-1, M).  Totals: all / attributed
// time, attributed and matched kernel counts.  Whether every kernel's row is
// its own index (the match of a trace whose ncu rows follow the kernels one
// for one) is noted, so the ops pass can skip the row-index gather; with
// ident_rows (a join whose matching was that identity pairing) the row
// indices are known to be the kernel indices and are not read.  Each
// attributed kernel (valid range and op id) also takes its slot among its
// op's kernels: one atomic per distinct op id of a warp on cnt[op], whose old
// value plus the kernel's rank among its warp peers is the slot (rank[k]);
// cnt ends as the per-op counts.  Each warp takes a run of `run` consecutive
// kernels (a multiple of 32, up to AF_RUN) in index order, so an op whose
// kernels all lie in one run gets ascending slots; the ops pass sorts the few
// segments that do not.
//
// Bound by the latency of the gathers and atomics of a step, so AC_GROUPS
// groups of 32 kernels go together: 116 us for 20M kernels, 264 for 50M (143
// and 409 one group at a time with its loads a step ahead; two groups 142 and
// 415, four with the registers of AC_BLOCKS blocks spilling 114 and 254, four
// with a block fewer 124 and 260).
constexpr int AF_RUN = 4096;
constexpr int AC_GROUPS = 3, AC_BLOCKS = 5;
constexpr int AC_PER = 16;                      // counts that a thread of the last block scans
constexpr int64_t AC_SCAN = 256 * AC_PER;

template <bool DIRECT>
__global__ void __launch_bounds__(256, AC_BLOCKS)
    k_agg_count(const int64_t *__restrict__ dur, const int32_t *__restrict__ rok, const int32_t *__restrict__ nidx,
                const uint32_t *__restrict__ r_op, int64_t K, int64_t R, int64_t M, int64_t n_ops,
                uint32_t *cnt, uint32_t *__restrict__ rank, int64_t run, int ident_rows,
                unsigned *__restrict__ nonident, int pending, uint32_t *off, unsigned *done, DevStatus *st) {
    pdl_wait();
    if (pending && stopped(st)) return;
    const unsigned lane = lane_id(), lt = lanemask_lt();
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
    const int64_t nwarps = (int64_t)gridDim.x * blockDim.x / 32;
    unsigned long long tot = 0, att = 0;
    unsigned natt = 0, nmatch = 0;
    int bad = 0, nid = 0;
    for (int64_t k0 = warp * run; k0 < K; k0 += nwarps * run) {
        const int64_t k1 = k0 + run < K ? k0 + run : K;
        for (int64_t kb = k0; kb < k1; kb += 32 * AC_GROUPS) {
            int32_t r[AC_GROUPS], j[AC_GROUPS];
            long long d[AC_GROUPS];
            uint32_t op[AC_GROUPS];
            unsigned peers[AC_GROUPS], base[AC_GROUPS];
            // the sums of a call with a bad record are not given out, so no
            // record waits for its checks
#pragma unroll
            for (int u = 0; u < AC_GROUPS; ++u) {
                const int64_t k = kb + u * 32 + lane;
                const bool in = k < k1;
                r[u] = in ? range_of_t<DIRECT>(rok, r_op, k) : -1;
                d[u] = in ? dur[k] : 0;
                j[u] = in ? (ident_rows ? (int32_t)k : nidx[k]) : -1;
            }
#pragma unroll
            for (int u = 0; u < AC_GROUPS; ++u) op[u] = (r[u] >= 0 && r[u] < R) ? r_op[r[u]] : 0xFFFFFFFFu;
#pragma unroll
            for (int u = 0; u < AC_GROUPS; ++u) {
                const int64_t k = kb + u * 32 + lane;
                nid |= k < k1 && (int64_t)j[u] != k;
                bad |= d[u] < 0 || r[u] < -1 || r[u] >= R || j[u] < -1 || j[u] >= M;
                tot += (unsigned long long)d[u];
                if (r[u] >= 0) {
                    att += (unsigned long long)d[u];
                    natt++;
                    nmatch += j[u] >= 0;
                    bad |= (int64_t)op[u] >= n_ops;
                }
                // slotted exactly as k_agg_place places it: by range and op id alone
                if ((int64_t)op[u] >= n_ops) op[u] = 0xFFFFFFFFu;
                peers[u] = __match_any_sync(0xffffffffu, op[u]);
                base[u] = 0;
                if (op[u] != 0xFFFFFFFFu && (peers[u] & lt) == 0) base[u] = atomicAdd(&cnt[op[u]], (unsigned)__popc(peers[u]));
            }
#pragma unroll
            for (int u = 0; u < AC_GROUPS; ++u) {
                base[u] = __shfl_sync(0xffffffffu, base[u], __ffs(peers[u]) - 1);
                if (op[u] != 0xFFFFFFFFu) rank[kb + u * 32 + lane] = base[u] + __popc(peers[u] & lt);
            }
        }
    }
    __shared__ unsigned long long red[33];
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_err(st, ERR_INVALID);
    if (__any_sync(0xffffffffu, nid) && lane_id() == 0) atomicOr(nonident, 1u);
    block_add_u64(tot, &st->cnt[C_TOTAL_NS], red);
    block_add_u64(att, &st->cnt[C_ATTR_NS], red);
    block_add_u64((unsigned long long)natt, &st->cnt[C_ATTR_K], red);
    block_add_u64((unsigned long long)nmatch, &st->cnt[C_MATCHED_K], red);
    if (!off) return;
    // few ops: the last block turns the counts into offsets
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    const int64_t i0 = threadIdx.x * AC_PER;
    uint32_t v[AC_PER], sum = 0;
#pragma unroll
    for (int i = 0; i < AC_PER; ++i) v[i] = i0 + i <= n_ops ? __ldcg(cnt + i0 + i) : 0u;
#pragma unroll
    for (int i = 0; i < AC_PER; ++i) sum += v[i];
    uint32_t ex = block_exclusive_scan<uint32_t>(sum, reinterpret_cast<uint32_t *>(red), nullptr);
#pragma unroll
    for (int i = 0; i < AC_PER; ++i) {
        if (i0 + i <= n_ops) off[i0 + i] = ex;
        ex += v[i];
    }
}

// ------------------------------------------------------------------ place
// list[off[op] + rank[k]] = k for each kernel k_agg_count slotted.
template <bool DIRECT>
__global__ void k_agg_place(const int32_t *__restrict__ rok, const uint32_t *__restrict__ r_op, int64_t K, int64_t R,
                            int64_t n_ops, const uint32_t *__restrict__ off, const uint32_t *__restrict__ rank,
                            uint32_t *__restrict__ list, int pending, const DevStatus *st) {
    pdl_wait();
    if (pending && stopped(st)) return;
    constexpr int U = 4;                    // kernels per thread per round, loads issued together
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t k0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k0 < K; k0 += stride * U) {
        int32_t r[U];
        uint32_t op[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = k0 + u * stride;
            r[u] = k < K ? range_of_t<DIRECT>(rok, r_op, k) : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) op[u] = (r[u] >= 0 && r[u] < R) ? r_op[r[u]] : 0xFFFFFFFFu;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t k = k0 + u * stride;
            if (r[u] >= 0 && r[u] < R && (int64_t)op[u] < n_ops) list[off[op[u]] + rank[k]] = (uint32_t)k;
        }
    }
}

// ------------------------------------------------------------------ long segments
// Segments of the ops longer than AG_MID_MAX (the pieces pass below), when a
// counting pass cannot place them in order, are sorted by kernel index first,
// one block per segment: up to SL_SMEM entries by a bitonic sort in shared
// memory; longer ones in SL_SMEM runs sorted that way, then merged pairwise
// through `tmp` (merge path: each thread merges an equal share of the output
// after a binary search on its diagonal).
constexpr int SL_THREADS = 256;
constexpr int SL_SMEM = 8192;

// Ops up to this length, or up to four times the average one, are left to one
// lane of the ops pass; AG_LANE_TOP at most.  4M kernels, ops of 200 in order /
// in any order / of skewed lengths: 743 / 869 / 1,157 us with 128 at most, where
// 256 took 2,387 / 3,294 / 2,032 (few lanes at work, each sorting by itself); ops
// of 100 in order 648, where 64 for all took 1,113.
constexpr uint32_t AG_LANE_MAX = 64, AG_LANE_TOP = 128;
constexpr uint32_t AG_MID_MAX = 4096;           // up to this length: one block; longer: pieces over several warps
constexpr uint32_t AG_PIECE = 1024;             // kernels of such an op per warp of the pieces pass

__device__ void bitonic_smem(uint32_t *a, int n2) {     // n2 a power of two; the block sorts a[0..n2)
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int q = threadIdx.x; q < n2 / 2; q += blockDim.x) {
                const int i = 2 * q - (q & (j - 1)), p = i + j;
                const uint32_t x = a[i], y = a[p];
                if (((i & k) == 0) == (x > y)) { a[i] = y; a[p] = x; }
            }
            __syncthreads();
        }
}

__global__ void __launch_bounds__(SL_THREADS) k_agg_sort_long(const uint32_t *__restrict__ off,
                                                              const uint32_t *__restrict__ longs,
                                                              const unsigned *__restrict__ nlong, uint32_t min_len,
                                                              uint32_t max_len, uint32_t *list, uint32_t *tmp) {
    pdl_wait();
    __shared__ uint32_t a[SL_SMEM];
    const unsigned n_long = *nlong;
    for (unsigned li = blockIdx.x; li < n_long; li += gridDim.x) {
        const uint32_t o = longs[li], s0 = off[o], len = off[o + 1] - s0;
        if (len < min_len || len > max_len) continue;      // uniform per block
        uint32_t *seg = list + s0, *alt = tmp + s0;
        // runs of SL_SMEM (the whole segment if it fits)
        for (uint32_t r0 = 0; r0 < len; r0 += SL_SMEM) {
            const int n = (int)(len - r0 < (uint32_t)SL_SMEM ? len - r0 : (uint32_t)SL_SMEM);
            int n2 = 1;
            while (n2 < n) n2 <<= 1;
            for (int i = threadIdx.x; i < n2; i += SL_THREADS) a[i] = i < n ? seg[r0 + i] : 0xFFFFFFFFu;
            __syncthreads();
            bitonic_smem(a, n2);
            for (int i = threadIdx.x; i < n; i += SL_THREADS) seg[r0 + i] = a[i];
            __syncthreads();
        }
        // merge passes, seg -> alt -> seg ...
        uint32_t *src = seg, *dst = alt;
        for (uint32_t w = SL_SMEM; w < len; w <<= 1) {
            for (uint32_t lo = 0; lo < len; lo += 2 * w) {
                const uint32_t mid = lo + w < len ? lo + w : len, hi = lo + 2 * w < len ? lo + 2 * w : len;
                const uint32_t na = mid - lo, nb = hi - mid, total = na + nb;
                const uint32_t share = (total + SL_THREADS - 1) / SL_THREADS;
                const uint32_t d0 = threadIdx.x * share < total ? threadIdx.x * share : total;
                const uint32_t d1 = d0 + share < total ? d0 + share : total;
                // i = items taken from run a among the first d0 outputs
                uint32_t ilo = d0 > nb ? d0 - nb : 0, ihi = d0 < na ? d0 : na;
                while (ilo < ihi) {
                    const uint32_t i = (ilo + ihi) >> 1;
                    if (src[lo + i] <= src[mid + (d0 - i - 1)]) ilo = i + 1; else ihi = i;
                }
                uint32_t i = ilo, j = d0 - ilo;
                for (uint32_t d = d0; d < d1; ++d) {
                    const bool take_a = j >= nb || (i < na && src[lo + i] <= src[mid + j]);
                    dst[lo + d] = take_a ? src[lo + i++] : src[mid + j++];
                }
            }
            __syncthreads();
            uint32_t *t = src; src = dst; dst = t;
        }
        if (src != seg) {
            for (uint32_t i = threadIdx.x; i < len; i += SL_THREADS) seg[i] = src[i];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------ ops
// One thread per op id.  Each warp takes AG_CHUNK consecutive op ids at a
// time, orders them by segment length (longest first) and walks them in
// AG_CHUNK / 32 rounds, so that the threads of a round walk segments of
// similar length and finish together (the record is written by every lane of
// the round at once); warps share nothing and never wait for each other.
// The grid is what stays resident; warps draw the chunks in increasing order
// from one counter (the next chunk is drawn, and its offsets loaded, while
// the current one runs), so the ops in flight at any moment are one narrow
// band of op ids whatever each warp's pace, and with op ids in range order
// the kernels and outputs of that band stay in L2.  The chunk's segments are
// one contiguous run of the list; when it fits it is first copied to shared
// memory, and each thread checks its segments there and,
// in the rare case the count pass met an op in two runs, sorts them in place,
// so segments are walked in ascending kernel index (a larger chunk reads the
// list in place).  Ops longer than lane_max are listed instead, for a block
// each or for the pieces pass: a lane waits up to a microsecond for each of its
// kernels, and one op of 250 held the pass (4M kernels with fusion operators:
// 589 us) for four times as long as all the others.  While a kernel is added,
// the counter rows and durations of the next two arrive in per-thread
// shared-memory slots by asynchronous copy (cp.async), with their row indices
// loaded a step earlier still (or taken to be the kernel indices when the count
// pass found every row to be its kernel's own index).
constexpr int AG_THREADS = 128;
constexpr int AG_WARPS = AG_THREADS / 32;
constexpr int AG_CHUNK = 64;                   // op ids per warp and chunk, at most
constexpr int AG_LBUCKETS = 32;
// Four blocks of four warps per multiprocessor, 656 us on 20M kernels and 340 on
// 6M whose records were out of order: with the 96 registers of five the
// accumulators spill (821 and 475), three measured slower too (as did four
// slots).  Chunks of 128 ops fill more lanes (49 % of them for 35 with a long
// tail of lengths) but put twice the ops in flight, past what L2 holds: 896 and 466.
// The chunk's offsets lie in shared memory and its list run comes by asynchronous
// copy; with the offsets in registers, handed round by shuffles, and the run copied
// through them, 704 and 345.
constexpr int AG_SLOTS = 2, AG_BLOCKS = 4;
constexpr int AG_STAGE = 1024;                  // list entries of a chunk staged in shared memory

struct OpsWarp {
    float4 row[AG_SLOTS][32][NC / 4];      // kernels in flight per thread: counter rows
    long long dur[AG_SLOTS][32];           // and durations, by asynchronous copy
    uint32_t L[AG_STAGE];           // the chunk's list run (when it fits)
    uint32_t off[2][AG_CHUNK + 4];  // the chunk's offsets (one more than ops), and the next one's
    uint32_t lcount[AG_LBUCKETS];
    uint8_t order[AG_CHUNK];
};
constexpr size_t AG_SMEM = sizeof(OpsWarp) * AG_WARPS;

// Ascending order of a segment of at most AG_LANE_TOP, sorted in place when it is
// not.  An op whose kernels lie in one run of the count pass is in order; in two
// neighbouring ones, two ascending runs, which insertion takes in one pass; one
// whose kernels lie anywhere, up to len^2 / 4 moves.
__device__ __forceinline__ void sort_segment(uint32_t *seg, uint32_t len) {
    bool up = true;
    for (uint32_t t = 1; t < len; ++t) up &= seg[t - 1] < seg[t];
    if (up) return;
    for (uint32_t t = 1; t < len; ++t) {
        const uint32_t x = seg[t];
        uint32_t u = t;
        for (; u > 0 && seg[u - 1] > x; --u) seg[u] = seg[u - 1];
        seg[u] = x;
    }
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The counter rows of a warp's 32 kernels to shared memory, dst[l] for lane l
// (row index j, -1 for none).  The lanes together copy 16-byte parts in the
// order they lie, so one copy instruction touches the seven rows its 512 bytes
// fall in, where each lane copying its own row touched 32 lines with every
// instruction and the L1's tag lookups bound the pass.  Every lane must call it;
// after the wait for its own copies a __syncwarp() makes the others' visible.
__device__ __forceinline__ void cp_async_rows(float4 (*dst)[NC / 4], const float4 *rows, int32_t j) {
    float4 *flat = &dst[0][0];
#pragma unroll
    for (int q = 0; q < NC / 4; ++q) {
        const unsigned e = q * 32 + lane_id(), r = e / (NC / 4), c = e - r * (NC / 4);
        const int32_t jr = __shfl_sync(0xffffffffu, j, (int)r);
        if (jr >= 0) cp_async16(flat + e, rows + (int64_t)jr * (NC / 4) + c);
    }
}

// Where the last block of the ops pass stores the status block and the numbers
// of listed ops for the host (mapped pinned memory), or NULL: a launch fewer
// before the host's wait.
struct OpsReport {
    uint32_t *status, *counts;
};

__global__ void __launch_bounds__(AG_THREADS, AG_BLOCKS) k_agg_ops(const uint32_t *__restrict__ off, uint32_t *list,
                                                          AggIn A, int pending, const DevStatus *st,
                                                          OpsReport report) {
    pdl_wait();
    const bool idle = pending && stopped(st);
    extern __shared__ __align__(16) unsigned char ag_smem[];
    OpsWarp &W = reinterpret_cast<OpsWarp *>(ag_smem)[threadIdx.x / 32];
    const unsigned lane = lane_id();
    const bool ident = *A.nonident == 0;
    const float4 *rows = reinterpret_cast<const float4 *>(A.counters);
    // row index of kernel k, -1 for none (or for an index past the rows)
    auto row_of = [&](uint32_t k) -> int32_t {
        const int32_t j = ident ? (int32_t)k : A.ncu_idx[k];
        return j < A.M ? j : -1;
    };
    auto draw = [&]() -> unsigned {
        unsigned v = 0;
        if (lane == 0) v = gridDim.x * AG_WARPS + atomicAdd(A.ctr, 1u);
        return v;
    };
    constexpr int PER = AG_CHUNK / 32;
    const int CHUNK = A.chunk;
    // the first chunk (each warp has one) and its offsets; afterwards the next
    // chunk is drawn and its offsets copied while the current one runs
    int64_t o0 = idle ? A.n_ops : (int64_t)(blockIdx.x * AG_WARPS + threadIdx.x / 32) * CHUNK;
    int buf = 0;
    auto fetch_offsets = [&](int to, int64_t o) {
        for (int i = (int)lane; i <= CHUNK && o + i <= A.n_ops; i += 32) cp_async4(&W.off[to][i], off + o + i);
        cp_async_commit();
    };
    if (o0 < A.n_ops) fetch_offsets(0, o0);
    cp_async_wait<0>();
    __syncwarp();
    while (o0 < A.n_ops) {
        const unsigned next_raw = draw();           // in flight during this chunk
        const int nchunk = A.n_ops - o0 < CHUNK ? (int)(A.n_ops - o0) : CHUNK;
        const uint32_t *offs = W.off[buf];
        const uint32_t cbase = offs[0], ctot = offs[nchunk] - cbase;       // the chunk's list run
        const bool staged = ctot <= AG_STAGE;
        // lengths of the chunk's ops, counting sort by length (descending, capped)
        uint32_t bkt[PER];
        W.lcount[lane] = 0;
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int i = q * 32 + (int)lane;
            const uint32_t len = i < nchunk ? offs[i + 1] - offs[i] : 0u;
            bkt[q] = AG_LBUCKETS - 1 - (len < AG_LBUCKETS - 1 ? len : AG_LBUCKETS - 1);
            if (i < nchunk) atomicAdd(&W.lcount[bkt[q]], 1u);
        }
        if (staged)
            for (uint32_t i = lane; i < ctot; i += 32) cp_async4(&W.L[i], list + cbase + i);
        cp_async_commit();
        __syncwarp();
        {
            const unsigned x = W.lcount[lane];
            const unsigned inc = warp_inclusive_scan(x);
            W.lcount[lane] = inc - x;
        }
        cp_async_wait<0>();
        __syncwarp();
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            const int i = q * 32 + (int)lane;
            if (i < nchunk) W.order[atomicAdd(&W.lcount[bkt[q]], 1u)] = (uint8_t)i;
            // each thread puts the segments of its own ops in ascending order
            const uint32_t len = i < nchunk ? offs[i + 1] - offs[i] : 0u;
            if (len > A.lane_max) {
                const bool mid = len <= AG_MID_MAX;
                (mid ? A.mids : A.longs)[atomicAdd(A.ctr + (mid ? 2 : 3), 1u)] = (uint32_t)(o0 + i);
            } else if (len > 1) {
                if (staged) sort_segment(W.L + (offs[i] - cbase), len);
                else sort_segment(list + offs[i], len);
            }
        }
        __syncwarp();
        // the next chunk's offsets, in flight during the rounds
        const int64_t o1 = (int64_t)__shfl_sync(0xffffffffu, next_raw, 0) * CHUNK;
        if (o1 < A.n_ops) fetch_offsets(buf ^ 1, o1);
        for (int g = 0; g * 32 < nchunk; ++g) {
            const int i = g * 32 + (int)lane;
            const int il = i < nchunk ? W.order[i] : 0;
            const uint32_t sa = offs[il], sb = offs[il + 1];
            const int64_t o = o0 + il;
            const bool mine = i < nchunk && sb - sa <= A.lane_max;             // (longer ones are listed)
            const uint32_t s0 = sa, len = mine ? sb - sa : 0u;
            const uint32_t most = __reduce_max_sync(0xffffffffu, len);         // the lanes copy rows together
            const uint32_t *seg = staged ? W.L + (s0 - cbase) : list + s0;
            AccF acc;
            acc.init();
            if (most > 0) {
                // kernel t's row and duration land in slot t % AG_SLOTS while the
                // kernels before it are added; row indices are loaded one step
                // further ahead
                auto issue = [&](uint32_t t, uint32_t k, int32_t j) {
                    if (t < len) cp_async8(&W.dur[t % AG_SLOTS][lane], A.dur + k);
                    cp_async_rows(W.row[t % AG_SLOTS], rows, j);
                    cp_async_commit();
                };
                unsigned have = 0;                    // bit t % AG_SLOTS: the kernel in that slot has a row
#pragma unroll
                for (uint32_t t = 0; t < (uint32_t)AG_SLOTS; ++t) {
                    const uint32_t kt = t < len ? seg[t] : 0u;
                    const int32_t jt = t < len ? row_of(kt) : -1;
                    issue(t, kt, jt);
                    have |= (jt >= 0 ? 1u : 0u) << t;
                }
                uint32_t k2 = AG_SLOTS < len ? seg[AG_SLOTS] : 0u;
                int32_t j2 = AG_SLOTS < len ? row_of(k2) : -1;
                for (uint32_t t = 0; t < most; ++t) {
                    const uint32_t k3 = t + AG_SLOTS + 1 < len ? seg[t + AG_SLOTS + 1] : 0u;
                    const int32_t j3 = t + AG_SLOTS + 1 < len ? row_of(k3) : -1;
                    cp_async_wait<AG_SLOTS - 1>();
                    __syncwarp();
                    const unsigned bit = 1u << (t % AG_SLOTS);
                    if (t < len) acc.accumulate(W.dur[t % AG_SLOTS][lane], have & bit, W.row[t % AG_SLOTS][lane]);
                    __syncwarp();
                    issue(t + AG_SLOTS, k2, j2);
                    have = j2 >= 0 ? have | bit : have & ~bit;
                    k2 = k3;
                    j2 = j3;
                }
                cp_async_wait<0>();
            }
            // a null or infinite value poisons a sum: the op is listed for
            // k_agg_careful
            if (!mine) continue;
            if (acc.clean()) acc.write(A, o, (int)len);
            else A.dirty[atomicAdd(A.ctr + 1, 1u)] = (uint32_t)o;
        }
        cp_async_wait<0>();
        __syncwarp();
        o0 = o1;
        buf ^= 1;
    }
    if (!report.status) return;
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(A.ctr + 4, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    for (unsigned i = threadIdx.x; i < sizeof(DevStatus) / 4; i += AG_THREADS)
        report.status[i] = __ldcg(reinterpret_cast<const uint32_t *>(st) + i);
    if (threadIdx.x < 3) report.counts[threadIdx.x] = __ldcg(A.ctr + 1 + threadIdx.x);
}

// The ops k_agg_ops listed as dirty: one lane each puts the segment in
// ascending kernel index (in place) and redoes it with AccN, which leaves
// nulls out and reports infinite values.  A separate pass keeps that
// register-hungry path out of the ops pass (within it, for the lanes concerned,
// the pass spilled: 853 us on 20M kernels without any null where it took 696).  Rows
// reach the lanes as they do there, the warp copying together and AG_SLOTS
// kernels ahead, counters two to a register.  Bound by issue at 12 warps a
// multiprocessor (1.6 instructions a cycle): 176,000 ops, 1M kernels with 2 % of
// nulls, 75 us; 86 with Acc and each lane reading its own rows.
__global__ void __launch_bounds__(AG_THREADS, AG_BLOCKS) k_agg_careful(const uint32_t *__restrict__ off,
                                                                       uint32_t *list, AggIn A, DevStatus *st) {
    pdl_wait();
    __shared__ float4 row_s[AG_WARPS][AG_SLOTS][32][NC / 4];
    __shared__ long long dur_s[AG_WARPS][AG_SLOTS][32];
    const unsigned lane = lane_id(), w = threadIdx.x / 32;
    auto &row = row_s[w];
    auto &dur = dur_s[w];
    const float4 *rows = reinterpret_cast<const float4 *>(A.counters);
    auto row_of = [&](uint32_t k) -> int32_t {
        const int32_t j = A.ncu_idx[k];
        return j < A.M ? j : -1;
    };
    int bad = 0;
    const unsigned n = A.ctr[1];
    for (unsigned e0 = (blockIdx.x * AG_WARPS + w) * 32; e0 < n; e0 += gridDim.x * AG_WARPS * 32) {
        const bool mine = e0 + lane < n;
        const uint32_t o = mine ? A.dirty[e0 + lane] : 0u;
        const uint32_t s0 = mine ? off[o] : 0u, len = mine ? off[o + 1] - s0 : 0u;
        const uint32_t most = __reduce_max_sync(0xffffffffu, len);
        uint32_t *seg = list + s0;
        sort_segment(seg, len);
        __syncwarp();
        auto issue = [&](uint32_t t, uint32_t k, int32_t j) {
            if (t < len) cp_async8(&dur[t % AG_SLOTS][lane], A.dur + k);
            cp_async_rows(row[t % AG_SLOTS], rows, j);
            cp_async_commit();
        };
        AccN acc;
        acc.init();
        unsigned have = 0;
#pragma unroll
        for (uint32_t t = 0; t < (uint32_t)AG_SLOTS; ++t) {
            const uint32_t kt = t < len ? seg[t] : 0u;
            const int32_t jt = t < len ? row_of(kt) : -1;
            issue(t, kt, jt);
            have |= (jt >= 0 ? 1u : 0u) << t;
        }
        uint32_t k2 = AG_SLOTS < len ? seg[AG_SLOTS] : 0u;
        int32_t j2 = AG_SLOTS < len ? row_of(k2) : -1;
        for (uint32_t t = 0; t < most; ++t) {
            const uint32_t k3 = t + AG_SLOTS + 1 < len ? seg[t + AG_SLOTS + 1] : 0u;
            const int32_t j3 = t + AG_SLOTS + 1 < len ? row_of(k3) : -1;
            cp_async_wait<AG_SLOTS - 1>();
            __syncwarp();
            const unsigned bit = 1u << (t % AG_SLOTS);
            if (t < len) acc.accumulate(dur[t % AG_SLOTS][lane], have & bit, row[t % AG_SLOTS][lane]);
            __syncwarp();
            issue(t + AG_SLOTS, k2, j2);
            have = j2 >= 0 ? have | bit : have & ~bit;
            k2 = k3;
            j2 = j3;
        }
        cp_async_wait<0>();
        __syncwarp();
        if (mine) {
            acc.write(A, o, (int)len);
            bad |= acc.bad;
        }
    }
    if (bad) set_err(st, ERR_INVALID);
}

// ------------------------------------------------------------------ host
// ------------------------------------------------------------------ long ops
// Ops longer than AG_MID_MAX that the ops pass lists (sorted by
// k_agg_sort_long or placed in order by a counting pass) are split into pieces
// of AG_PIECE kernels, so an operator with a very long segment (an Inductor
// fusion-map operator gathers every unattributed launch of its kernel name) is
// spread over many warps instead of holding one block for its whole length.
// Each lane adds a
// contiguous run of a piece in ascending kernel index with the careful
// accumulator; partials are combined by fixed trees of pairwise float-float
// additions (lane l takes lane l + 16, then l + 8, ...; a piece's partials in
// piece order), so results are reproducible, with an error bound of the
// longest run (32 kernels in a piece) plus the pairwise steps.
__device__ __forceinline__ ff ff_pair_add(ff a, ff b) {
    const ff t = two_sum(a.hi, b.hi);
    return ff{t.hi, __fadd_rn(t.lo, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ ff shfl_down_ff(ff v, int d) {
    return ff{__shfl_down_sync(0xffffffffu, v.hi, d), __shfl_down_sync(0xffffffffu, v.lo, d)};
}
__device__ __forceinline__ void acc_merge_down(Acc &a, int d) {
    const bool take = (int)lane_id() < d;
    const int kc = __shfl_down_sync(0xffffffffu, a.kc, d), mc = __shfl_down_sync(0xffffffffu, a.mc, d);
    const long long ds = __shfl_down_sync(0xffffffffu, a.dsum, d), da = __shfl_down_sync(0xffffffffu, a.dall, d);
    const unsigned seen = __shfl_down_sync(0xffffffffu, a.seen, d);
    const int bad = __shfl_down_sync(0xffffffffu, a.bad, d);
    if (take) {
        a.kc += kc; a.mc += mc; a.dsum += ds; a.dall += da; a.seen |= seen; a.bad |= bad;
    }
#pragma unroll
    for (int i = 0; i < N_SUM; ++i) {
        const ff x = shfl_down_ff(a.s[i], d);
        if (take) a.s[i] = ff_pair_add(a.s[i], x);
    }
#pragma unroll
    for (int i = 0; i < N_DW; ++i) {
        const ff x = shfl_down_ff(a.w[i], d);
        const long long nw = __shfl_down_sync(0xffffffffu, a.nanw[i], d);
        if (take) {
            a.w[i] = ff_pair_add(a.w[i], x);
            a.nanw[i] += nw;
        }
    }
#pragma unroll
    for (int i = 0; i < N_MAX; ++i) {
        const float x = __shfl_down_sync(0xffffffffu, a.mx[i], d);
        if (take) a.mx[i] = fmaxf(a.mx[i], x);
    }
}
// a += b, the same pairwise steps as acc_merge_down
__device__ __forceinline__ void acc_merge(Acc &a, const Acc &b) {
    a.kc += b.kc; a.mc += b.mc; a.dsum += b.dsum; a.dall += b.dall; a.seen |= b.seen; a.bad |= b.bad;
#pragma unroll
    for (int i = 0; i < N_SUM; ++i) a.s[i] = ff_pair_add(a.s[i], b.s[i]);
#pragma unroll
    for (int i = 0; i < N_DW; ++i) {
        a.w[i] = ff_pair_add(a.w[i], b.w[i]);
        a.nanw[i] += b.nanw[i];
    }
#pragma unroll
    for (int i = 0; i < N_MAX; ++i) a.mx[i] = fmaxf(a.mx[i], b.mx[i]);
}

// Piece offsets of the listed ops, one block: poff[j] = pieces of the ops listed
// before j (ceil(kernels / AG_PIECE) each); poff[number of them] = all pieces.
__global__ void __launch_bounds__(1024) k_agg_piece_offsets(const uint32_t *__restrict__ off,
                                                            const uint32_t *__restrict__ longs,
                                                            const unsigned *__restrict__ nlong,
                                                            uint32_t *__restrict__ poff) {
    pdl_wait();
    __shared__ uint32_t wbuf[33];
    const int64_t n = *nlong;
    uint32_t carry = 0;
    for (int64_t b = 0; b < n; b += 1024) {
        const int64_t j = b + threadIdx.x;
        uint32_t np = 0;
        if (j < n) {
            const uint32_t o = longs[j];
            np = (off[o + 1] - off[o] + AG_PIECE - 1) / AG_PIECE;
        }
        uint32_t tot;
        const uint32_t ex = block_exclusive_scan<uint32_t>(np, wbuf, &tot);
        if (j < n) poff[j] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) poff[n] = carry;
}

// Huge ops' segments in ascending kernel index without sorting: with at most
// 256 huge ops, one counting pass over all kernels in index order, the digit
// being the index of the kernel's op among the huge ops, writes each such
// kernel to its op's segment at its rank among the op's kernels.
struct HugeDigit {
    const int32_t *rok;
    const uint32_t *r_op;
    int64_t R, n_ops;
    const uint32_t *hidx;        // [n_ops] index of a huge op among the huge ops, else 0xFFFFFFFF
    __device__ __forceinline__ unsigned operator()(int64_t k) const {
        const int32_t r = range_of(rok, r_op, k);
        if (r < 0 || r >= R) return RADIX_BINS;
        const uint32_t op = r_op[r];
        if ((int64_t)op >= n_ops) return RADIX_BINS;
        const uint32_t j = hidx[op];
        return j < RADIX_BINS ? j : (unsigned)RADIX_BINS;
    }
};
struct HugePlace {
    const uint32_t *hist;        // scanned digit-major histogram: hist[j * ntiles] = start of digit j
    int64_t ntiles;
    const uint32_t *hop, *off;   // the huge ops; the segment offsets
    uint32_t *list;
    __device__ __forceinline__ unsigned operator()(int64_t k, uint32_t dest, unsigned j) const {
        list[off[hop[j]] + (dest - hist[(int64_t)j * ntiles])] = (uint32_t)k;
        return 0u;
    }
    __device__ __forceinline__ void done(unsigned) const {}
};
__global__ void k_huge_index(const uint32_t *__restrict__ hop, int64_t n_huge, uint32_t *__restrict__ hidx) {
    pdl_wait();
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n_huge; c += (int64_t)gridDim.x * blockDim.x)
        hidx[hop[c]] = (uint32_t)c;
}

// A fast partial in careful form (every counter of every matched kernel non-null).
__device__ __forceinline__ void acc_from_fast(Acc &out, const AccF &f, int kc) {
    out.kc = kc;
    out.mc = f.mc;
    out.dsum = f.dsum;
    out.dall = f.dall;
#pragma unroll
    for (int i = 0; i < N_SUM; ++i) out.s[i] = f.sum(Acc::sum_col(i));
#pragma unroll
    for (int i = 0; i < N_DW; ++i) {
        out.w[i] = f.sum(Acc::dw_col(i));
        out.nanw[i] = 0;
    }
#pragma unroll
    for (int i = 0; i < N_MAX; ++i) out.mx[i] = f.mx[i];
    out.seen = f.mc > 0 ? ALL_COUNTERS : 0u;
    out.bad = 0;
    out.terms = 0;
}
// A lane's run of a piece with the fast accumulator: returns false when a
// null or infinite value took part (the caller redoes the run carefully),
// else the run's partial in careful form (every counter non-null).
__device__ __forceinline__ bool piece_fast(const AggIn &A, const uint32_t *seg, uint32_t l0, uint32_t l1, Acc &out) {
    AccF f;
    f.init();
#pragma unroll 4
    for (uint32_t t = l0; t < l1; ++t) {
        const uint32_t k = seg[t];
        const int32_t j = A.ncu_idx[k];
        const bool ok = j >= 0 && j < A.M;
        f.accumulate(A.dur[k], ok, reinterpret_cast<const float4 *>(A.counters + (int64_t)(ok ? j : 0) * NC));
    }
    if (!f.clean()) return false;
    acc_from_fast(out, f, (int)(l1 - l0));
    return true;
}

// The same partial with the rows ahead: kernel t + PC_AHEAD's row and duration
// arrive in the lane's shared-memory slots by asynchronous copy while kernel t
// is added, its indices loaded two steps earlier still.  Every lane of the warp
// calls it.
constexpr int PC_SLOTS = 4, PC_AHEAD = PC_SLOTS - 1, PC_THREADS = 256;
struct PieceSlots {
    float4 row[PC_SLOTS][32][NC / 4];
    long long dur[PC_SLOTS][32];
};
constexpr size_t PC_SMEM = sizeof(PieceSlots) * (PC_THREADS / 32);
template <typename At>                       // at(t): the lane's t-th kernel, t < n
__device__ __forceinline__ bool piece_ahead(const AggIn &A, At at, uint32_t n, PieceSlots &S, Acc &out) {
    const unsigned lane = lane_id();
    const float4 *rows = reinterpret_cast<const float4 *>(A.counters);
    auto row_of = [&](uint32_t k) -> int32_t {
        const int32_t j = A.ncu_idx[k];
        return j < A.M ? j : -1;
    };
    auto issue = [&](uint32_t t, uint32_t k, int32_t j) {
        if (t < n) cp_async8(&S.dur[t % PC_SLOTS][lane], A.dur + k);
        cp_async_rows(S.row[t % PC_SLOTS], rows, j);
        cp_async_commit();
    };
    const uint32_t most = __reduce_max_sync(0xffffffffu, n);       // the lanes copy together
    AccF f;
    f.init();
    unsigned have = 0;                       // bit t % PC_SLOTS: the kernel in that slot has a row
    uint32_t k = 0;
    int32_t j = -1;
#pragma unroll
    for (uint32_t t = 0; t < (uint32_t)PC_AHEAD; ++t) {
        const uint32_t kt = t < n ? at(t) : 0u;
        const int32_t jt = t < n ? row_of(kt) : -1;
        issue(t, kt, jt);
        have |= (jt >= 0 ? 1u : 0u) << t;
    }
    if (PC_AHEAD < n) {
        k = at(PC_AHEAD);
        j = row_of(k);
    }
    uint32_t k2 = PC_AHEAD + 1 < n ? at(PC_AHEAD + 1) : 0u;
    for (uint32_t t = 0; t < most; ++t) {
        const int32_t j2 = t + PC_AHEAD + 1 < n ? row_of(k2) : -1;
        const uint32_t k3 = t + PC_AHEAD + 2 < n ? at(t + PC_AHEAD + 2) : 0u;
        cp_async_wait<PC_AHEAD - 1>();
        __syncwarp();
        if (t < n) f.accumulate(S.dur[t % PC_SLOTS][lane], (have >> (t % PC_SLOTS)) & 1u, S.row[t % PC_SLOTS][lane]);
        __syncwarp();
        issue(t + PC_AHEAD, k, j);
        const unsigned bit = 1u << ((t + PC_AHEAD) % PC_SLOTS);
        have = j >= 0 ? have | bit : have & ~bit;
        k = k2;
        j = j2;
        k2 = k3;
    }
    cp_async_wait<0>();
    if (!f.clean()) return false;
    acc_from_fast(out, f, (int)n);
    return true;
}

// A warp's kernels, n of them this lane's: the 32 partials merged by the fixed
// tree into *part.
template <typename At>
__device__ __forceinline__ void piece_by_warp(const AggIn &A, At at, uint32_t n, PieceSlots &S, Acc *part) {
    const uint32_t lane = lane_id();
    Acc acc;
    if (!piece_ahead(A, at, n, S, acc)) {                 // a null or infinite value: redo with null handling
        acc.init();
        for (uint32_t t = 0; t < n; ++t) acc.add(A, at(t));
    }
    __syncwarp();
#pragma unroll 1
    for (int d = 16; d > 0; d >>= 1) acc_merge_down(acc, d);
    if (lane == 0) *part = acc;
}

// Pieces: one warp per AG_PIECE kernels of a huge op, the piece's partial stored
// at its index.  Bound by the gathers of the rows (80 bytes in three or four
// sectors each).
__global__ void __launch_bounds__(PC_THREADS, 2) k_agg_pieces(const uint32_t *__restrict__ off, const uint32_t *__restrict__ list,
                             const uint32_t *__restrict__ longs, const unsigned *__restrict__ nlong,
                             const uint32_t *__restrict__ poff, AggIn A, Acc *__restrict__ part) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char ag_smem[];
    PieceSlots &S = reinterpret_cast<PieceSlots *>(ag_smem)[threadIdx.x / 32];
    const int64_t n = *nlong;
    const int64_t P = poff[n];
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t p = warp; p < P; p += nwarps) {
        int64_t lo = 0, hi = n;                   // the listed op: last j with poff[j] <= p
        while (hi - lo > 1) {
            const int64_t m = (lo + hi) >> 1;
            if ((int64_t)poff[m] <= p) lo = m; else hi = m;
        }
        const uint32_t o = longs[lo];
        const uint32_t s0 = off[o], len = off[o + 1] - s0;
        const uint32_t b0 = (uint32_t)(p - poff[lo]) * AG_PIECE;
        const uint32_t b1 = b0 + AG_PIECE < len ? b0 + AG_PIECE : len;
        const uint32_t *seg = list + s0 + b0;
        const uint32_t m = b1 - b0, per = (m + 31) / 32, l0 = min(lane_id() * per, m);   // consecutive shares
        piece_by_warp(A, [&](uint32_t t) { return seg[l0 + t]; }, min(l0 + per, m) - l0, S, part + p);
    }
}
static void launch_pieces(Ctx &c, const uint32_t *off, const uint32_t *list, const uint32_t *longs,
                          const unsigned *nlong, const uint32_t *poff, const AggIn &in, Acc *part) {
    cudaFuncSetAttribute(k_agg_pieces, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PC_SMEM);
    launch(c, "agg_pieces", k_agg_pieces, dim3(4 * sm_count(c)), dim3(PC_THREADS), PC_SMEM, off, list, longs, nlong,
           poff, in, part);
}

// Ops of more than lane_max and up to AG_MID_MAX kernels: a block each.  The
// segment comes to shared memory and is put in ascending kernel index when it is
// not; each thread adds a contiguous run of it, and the partials are merged by
// fixed trees (each warp's, then the warps' in order).  Two launches share the
// list: blocks of 128 threads take ops up to MID_SPLIT kernels, blocks of 512
// the longer ones (an op of 4,000 kernels takes 128 threads 250 us, most of it
// in the sort).
constexpr uint32_t MID_SPLIT = 1024;
template <int MID_THREADS>
__global__ void __launch_bounds__(MID_THREADS) k_agg_mid(const uint32_t *__restrict__ off,
                                                         const uint32_t *__restrict__ list, AggIn A, DevStatus *st) {
    pdl_wait();
    __shared__ uint32_t seg[AG_MID_MAX];
    __shared__ Acc wpart[MID_THREADS / 32];
    const unsigned lane = lane_id(), w = threadIdx.x >> 5, n = A.ctr[2];
    int bad = 0;
    for (unsigned q = blockIdx.x; q < n; q += gridDim.x) {
        const uint32_t o = A.mids[q], s0 = off[o], len = off[o + 1] - s0;
        if ((len > MID_SPLIT) != (MID_THREADS > 128)) continue;           // the other launch's
        uint32_t n2 = MID_THREADS;
        while (n2 < len) n2 <<= 1;
        bool down = false;
        for (uint32_t i = threadIdx.x; i < n2; i += MID_THREADS) {
            const uint32_t x = i < len ? list[s0 + i] : 0xFFFFFFFFu;
            down |= i + 1 < len && list[s0 + i + 1] < x;
            seg[i] = x;
        }
        if (__syncthreads_or(down)) bitonic_smem(seg, (int)n2);
        const uint32_t per = (len + MID_THREADS - 1) / MID_THREADS;
        const uint32_t l0 = min(threadIdx.x * per, len), l1 = min(l0 + per, len);
        Acc acc;
        if (!piece_fast(A, seg, l0, l1, acc)) {           // a null or infinite value: redo with null handling
            acc.init();
            for (uint32_t t = l0; t < l1; ++t) acc.add(A, seg[t]);
        }
#pragma unroll 1
        for (int d = 16; d > 0; d >>= 1) acc_merge_down(acc, d);
        if (lane == 0) wpart[w] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            Acc total = wpart[0];
            for (int v = 1; v < MID_THREADS / 32; ++v) acc_merge(total, wpart[v]);
            total.write(A, o);
            bad |= total.bad;
        }
        __syncthreads();
    }
    if (bad) set_err(st, ERR_INVALID);
}

// Finish: one block per huge op merges its pieces' partials -- thread t takes
// pieces t, t + FIN_THREADS, ... in order, then each warp's fixed tree, then
// thread 0 takes the warps' partials in warp order -- and writes the record.
constexpr int FIN_THREADS = 256;
__global__ void __launch_bounds__(FIN_THREADS) k_agg_long_ops(const uint32_t *__restrict__ longs,
                                                              const unsigned *__restrict__ nlong,
                                                              const uint32_t *__restrict__ poff,
                                                              const Acc *__restrict__ part, AggIn A,
                                                              DevStatus *st) {
    pdl_wait();
    __shared__ Acc wpart[FIN_THREADS / 32];
    const int64_t n = *nlong;
    const unsigned lane = lane_id(), w = threadIdx.x >> 5;
    int bad = 0;
    for (int64_t q = blockIdx.x; q < n; q += gridDim.x) {
        const uint32_t o = longs[q];
        Acc acc;
        acc.init();
        for (uint32_t p = poff[q] + threadIdx.x; p < poff[q + 1]; p += FIN_THREADS) acc_merge(acc, part[p]);
#pragma unroll 1
        for (int d = 16; d > 0; d >>= 1) acc_merge_down(acc, d);
        if (lane == 0) wpart[w] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            Acc total = wpart[0];
            for (int v = 1; v < FIN_THREADS / 32; ++v) acc_merge(total, wpart[v]);
            total.write(A, o);
            bad |= total.bad;
        }
        __syncthreads();
    }
    if (bad) set_err(st, ERR_INVALID);
}

// Blocks of the ops pass: what stays resident, fewer for few ops.  A chunk is
// half as long where every warp still has one at most: a lane then walks one op
// instead of two (14,300 ops 20 us -> 11; 114,400 ops, past that line, 23 us
// with chunks of 64).
static unsigned ops_grid(Ctx &c, int64_t O, int *chunk) {
    const int sms = sm_count(c);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_agg_ops, AG_THREADS, AG_SMEM);
    cudaGetLastError();
    const int64_t resident = (int64_t)std::max(1, sms) * std::max(1, per_sm);
    *chunk = O <= resident * AG_WARPS * (AG_CHUNK / 2) ? AG_CHUNK / 2 : AG_CHUNK;
    const int64_t need = (O + (int64_t)AG_WARPS * *chunk - 1) / ((int64_t)AG_WARPS * *chunk);
    return (unsigned)std::max<int64_t>(1, std::min(resident, need));
}

int64_t agg_counter_words(uint32_t n_ops) {
    const int64_t n = (int64_t)n_ops + 1;
    return AGG_OWN_WORDS + (scan_clean_words(n) + 7) / 8 * 8 + n;
}

// Ops longer than a lane takes, at most; pieces of the longest.
static int64_t agg_mids(int64_t K, int64_t O) { return std::min<int64_t>(O, K / (AG_LANE_MAX + 1)) + 1; }
static int64_t agg_partials(int64_t K) { return K / AG_PIECE + K / (AG_MID_MAX + 1) + 1; }
size_t aggregate_scratch(int64_t K, uint32_t n_ops) {
    const int64_t O = n_ops, mids_n = agg_mids(K, O);
    Need nd;
    nd.add<uint32_t>(O + 1).add<uint32_t>(K).add<uint32_t>(K);
    nd.add<uint32_t>(mids_n).add<uint32_t>(mids_n).add<uint32_t>(O + 1);
    nd.add<uint32_t>(mids_n).add<Acc>(agg_partials(K));
    nd.add<uint32_t>(scan_scratch_elems(std::max<int64_t>(O + 1, radix_hist_elems(K))));
    nd.add<uint32_t>(O + 1).add<uint32_t>(radix_hist_elems(K));       // huge-op index, histogram
    return nd.bytes + 4096;
}

opattr_status do_aggregate(Ctx &c, const opattr_kernels *kern, const opattr_ranges *rng, const int32_t *rok,
                           const opattr_ncu *ncu, const int32_t *nidx, uint32_t n_ops,
                           const opattr_op_aggregates *out, opattr_totals *tot_out) {
    const int64_t K = kern->n, R = rng->n, M = ncu->n, O = n_ops;
    if (K < 0 || R < 0 || M < 0 || K >= (1ll << 31) || R >= (1ll << 31) || M >= (1ll << 31) || !out)
        return OPATTR_E_INVALID_ARG;
    if (K > 0 && (!kern->dur_ns || !nidx)) return OPATTR_E_INVALID_ARG;
    if (K > 0 && !rok && R != K) return OPATTR_E_INVALID_ARG;     // one operator per kernel in rng->op_id
    if (R > 0 && !rng->op_id) return OPATTR_E_INVALID_ARG;
    if (M > 0 && !ncu->counters) return OPATTR_E_INVALID_ARG;
    if (O > 0 && (!out->kernel_count || !out->total_duration_ns || !out->matched_count || !out->agg))
        return OPATTR_E_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(ncu->counters) & 15) != 0) return OPATTR_E_INVALID_ARG;

    const int64_t mids_n = agg_mids(K, O), part_n = agg_partials(K);
    const size_t need = aggregate_scratch(K, n_ops);
    // the counters lie ready at the start of the arena, or are taken and zeroed here
    const int64_t words = agg_counter_words(n_ops);          // ctr, the scan's, cnt
    const bool keeps = c.enclose_pending || c.keep_status;
    if (!(keeps && c.agg_words == words)) c.agg_ready = false;
    if (!c.agg_ready) c.arena_keep = 0;
    opattr_status st = ensure_arena(c, need);
    if (!st && !c.agg_ready) st = ensure_arena(c, need + Need().add<uint32_t>(words).bytes);
    if (st) return st;
    Arena a(c);
    const bool ready = c.agg_ready;
    uint32_t *counters = ready ? reinterpret_cast<uint32_t *>(c.arena) : a.take<uint32_t>(words);
    c.agg_ready = false;
    c.arena_keep = 0;
    uint32_t *off = a.take<uint32_t>(O + 1);
    // tmp holds each kernel's slot among its op's kernels until the list is
    // placed, then serves the segment sorts
    uint32_t *list = a.take<uint32_t>(K), *tmp = a.take<uint32_t>(K);
    uint32_t *mids = a.take<uint32_t>(mids_n), *longs = a.take<uint32_t>(mids_n);
    // the numbers of ops listed dirty, mid and long (nlong) come back together
    if (!counters) return OPATTR_E_OOM;
    unsigned *ctr = counters, *nlong = ctr + 3, *nonident = ctr + 5;
    uint32_t *chain = counters + AGG_OWN_WORDS, *cnt = counters + (words - (O + 1));
    uint32_t *dirty = a.take<uint32_t>(O + 1);
    uint32_t *npc = a.take<uint32_t>(mids_n);
    Acc *partials = a.take<Acc>(part_n);
    if (!npc || !partials) return OPATTR_E_OOM;
    uint32_t *part = a.take<uint32_t>(scan_scratch_elems(std::max<int64_t>(O + 1, radix_hist_elems(K))));
    uint32_t *hidx = a.take<uint32_t>(O + 1), *hhist = a.take<uint32_t>(radix_hist_elems(K));
    if (!hidx || !hhist) return OPATTR_E_OOM;
    if (!off || !list || !tmp || !mids || !longs || !part || !dirty) return OPATTR_E_OOM;
    // with the enclosure's or the matching's verdict pending (a join) the status
    // block keeps it: the enclosure's reset left the aggregation's slots at zero
    const ZeroRun zr{counters, words};
    if (!ready && (st = keeps ? zero_runs(c, 1, &zr) : reset_status(c, 1, &zr))) return st;
    const int sms = sm_count(c);
    // Fewer than AC_SCAN ops: the count's last block scans the counts (340 ops:
    // 2 us more in the count, where the launch of a scan took 5); with 7,150 it
    // takes 8 us more, with 14,300 14 us, and one block of 1,024 threads 5 to 6.
    const bool scan = K > 0 && O > 0 && O < AC_SCAN;
    // runs long enough to keep most segments in one warp, in as few full waves
    // of resident warps as runs of up to AF_RUN allow
    const int64_t warps = (int64_t)std::max(1, sms) * AC_BLOCKS * 8, waves = (K + warps * AF_RUN - 1) / (warps * AF_RUN);
    const int64_t run = std::max<int64_t>(32, waves > 0 ? ((K + warps * waves - 1) / (warps * waves) + 31) / 32 * 32 : 0);
    if (K > 0)
        launch(c, "agg_count", rok ? k_agg_count<false> : k_agg_count<true>,
               dim3(grid_for(K, 256 / 32 * run, 65535)), dim3(256), 0, kern->dur_ns, rok, nidx, rng->op_id, K, R, M,
               O, cnt, tmp, run, (int)(c.in_join && c.rows_identity), nonident, (int)c.enclose_pending, scan ? off : nullptr,
               ctr + 6, c.d_status);
    AggIn in;
    in.dur = kern->dur_ns;
    in.ncu_idx = nidx;
    in.counters = ncu->counters;
    in.M = M;
    in.n_ops = O;
    in.lane_max = (uint32_t)std::min<int64_t>(AG_LANE_TOP, std::max<int64_t>(AG_LANE_MAX, O > 0 ? 4 * K / O : 0));
    in.ctr = ctr;
    in.dirty = dirty;
    in.mids = mids;
    in.longs = longs;
    in.nonident = nonident;
    in.out = *out;
    bool status_fresh = false;        // no launch since the last status read
    if (O > 0) {
        if (!scan) scan_exclusive_u32(c, cnt, off, O + 1, chain, nullptr, true);
        if (K > 0)
            launch(c, "agg_place", rok ? k_agg_place<false> : k_agg_place<true>,
                   dim3(grid_for(K, 256 * 4, REDUCE_GRID)), dim3(256), 0, rok, rng->op_id, K, R, O,
                   (const uint32_t *)off, (const uint32_t *)tmp, list, (int)c.enclose_pending,
                   (const DevStatus *)c.d_status);
        static unsigned attr_done = 0;
        if (c.device < 32 && !(attr_done & (1u << c.device))) {
            cudaFuncSetAttribute(k_agg_ops, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AG_SMEM);
            attr_done |= 1u << c.device;
        }
        const unsigned grid = ops_grid(c, O, &in.chunk);
        OpsReport report{};
        if (c.host_mapped) report = {reinterpret_cast<uint32_t *>(c.h_status), c.h_small};
        launch(c, "agg_ops", k_agg_ops, dim3(grid), dim3(AG_THREADS), AG_SMEM, (const uint32_t *)off, list, in,
               (int)c.enclose_pending, (const DevStatus *)c.d_status, report);
        // the ops the pass left: listed with a null or infinite value (redone
        // by k_agg_careful, a lane each), longer than a lane takes (a block
        // each) and longer still (the pieces pass); the counts come back with
        // the status
        const SmallCopy counts{c.h_small, ctr + 1, 3 * sizeof(uint32_t)};
        if ((st = c.host_mapped ? sync_status(c) : read_status(c, 1, &counts))) return st;
        const uint32_t n_dirty = c.h_small[0], n_mid = c.h_small[1], n_long = c.h_small[2];
        status_fresh = n_dirty == 0 && n_mid == 0 && n_long == 0;
        if (n_dirty > 0)
            launch(c, "agg_careful", k_agg_careful, dim3(grid_for(n_dirty, AG_THREADS)), dim3(AG_THREADS), 0,
                   (const uint32_t *)off, list, in, c.d_status);
        if (n_mid > 0) {
            launch(c, "agg_mid", k_agg_mid<128>, dim3(std::min<uint32_t>(n_mid, 4u * sms)), dim3(128), 0,
                   (const uint32_t *)off, (const uint32_t *)list, in, c.d_status);
            launch(c, "agg_mid", k_agg_mid<512>, dim3(std::min<uint32_t>(n_mid, (unsigned)sms)), dim3(512), 0,
                   (const uint32_t *)off, (const uint32_t *)list, in, c.d_status);
        }
        if (n_long > 0) {
            launch(c, "agg_piece_offsets", k_agg_piece_offsets, dim3(1), dim3(1024), 0, (const uint32_t *)off,
                   (const uint32_t *)longs, (const unsigned *)nlong, npc);
            if (n_long <= (uint32_t)RADIX_BINS) {
                // very long segments: placed in kernel order by one counting pass
                cudaMemsetAsync(hidx, 0xFF, sizeof(uint32_t) * (O + 1), c.stream);
                launch(c, "huge_index", k_huge_index, dim3(grid_for(n_long, 256, 4096)), dim3(256), 0,
                       (const uint32_t *)longs, (int64_t)n_long, hidx);
                const HugeDigit dg{rok, rng->op_id, R, O, hidx};
                const uint32_t *hoffs = digit_offsets(c, dg, K, hhist, part);
                const int64_t ntiles = (K + RADIX_TILE - 1) / RADIX_TILE;
                digit_rank(c, "huge_place", dg, K, hoffs,
                           HugePlace{hoffs, ntiles, (const uint32_t *)longs, (const uint32_t *)off, list});
            } else {
                launch(c, "agg_sort_long", k_agg_sort_long, dim3(2 * std::max(1, sms)), dim3(SL_THREADS), 0,
                       (const uint32_t *)off, (const uint32_t *)longs, (const unsigned *)nlong, 2u,
                       0xFFFFFFFFu, list, tmp);
            }
            launch_pieces(c, off, list, longs, nlong, npc, in, partials);
            launch(c, "agg_long_ops", k_agg_long_ops, dim3(2 * std::max(1, sms)), dim3(FIN_THREADS), 0,
                   (const uint32_t *)longs, (const unsigned *)nlong, (const uint32_t *)npc,
                   (const Acc *)partials, in, c.d_status);
        }
    }
    if (!status_fresh && (st = read_status(c))) return st;
    if (c.h_status->err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
    opattr_totals T{};
    T.total_ns = (int64_t)c.h_status->cnt[C_TOTAL_NS];
    T.attributed_ns = (int64_t)c.h_status->cnt[C_ATTR_NS];
    T.unattributed_ns = T.total_ns - T.attributed_ns;
    T.kernels = K;
    T.attributed_kernels = (int64_t)c.h_status->cnt[C_ATTR_K];
    T.matched_kernels = (int64_t)c.h_status->cnt[C_MATCHED_K];
    const double qnan = __builtin_nan("");
    T.attributed_frac = T.total_ns > 0 ? (double)T.attributed_ns / (double)T.total_ns : qnan;
    T.unattributed_frac = T.total_ns > 0 ? (double)T.unattributed_ns / (double)T.total_ns : qnan;
    if (tot_out) *tot_out = T;
    return OPATTR_OK;
}

}  // namespace opattr

namespace opattr {

// ------------------------------------------------------------------ class roll-up
// The per-operator records of Eq. (1) rolled up to operator classes (the
// per-class breakdown of the case studies): every attributed kernel whose
// operator has a class is aggregated with the other kernels of that class.
// Few, large groups, the kernels in index order within each: up to CLASS_DIGIT
// classes are grouped by one counting pass and summed by all warps of one wave,
// each on a share of one class (k_class_sums); more classes go through a stable
// radix sort by class key and the pieces of the long operators.
__global__ void k_class_check(const uint32_t *__restrict__ class_of_op, int64_t n_ops, uint32_t n_classes,
                              DevStatus *st) {
    pdl_wait();
    int bad = 0;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < n_ops; o += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t c = class_of_op[o];
        bad |= c >= n_classes && c != OPATTR_OP_NONE;
    }
    if (__any_sync(0xffffffffu, bad) && lane_id() == 0) set_err(st, ERR_INVALID);
}
// key = class of the kernel's operator, n_classes when it has none; counts
// per class (in a block histogram in shared memory when there are at most
// CK_SMEM classes, flushed once per block; else one global atomic per class
// and warp).
constexpr int CK_SMEM = 4096;
__global__ void k_class_keys(const int32_t *__restrict__ rok, const uint32_t *__restrict__ r_op, int64_t K, int64_t R,
                             int64_t n_ops, const uint32_t *__restrict__ class_of_op, uint32_t n_classes,
                             uint32_t *__restrict__ key, uint32_t *__restrict__ cnt) {
    pdl_wait();
    __shared__ uint32_t h[CK_SMEM];
    const bool local = n_classes <= (uint32_t)CK_SMEM;
    if (local)
        for (uint32_t i = threadIdx.x; i < n_classes; i += blockDim.x) h[i] = 0;
    __syncthreads();
    uint32_t *dst = local ? h : cnt;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k - threadIdx.x < K;
         k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t c = n_classes;
        if (k < K) {
            const int32_t r = range_of(rok, r_op, k);
            if (r >= 0 && r < R) {
                const uint32_t op = r_op[r];
                if ((int64_t)op < n_ops) {
                    const uint32_t x = class_of_op[op];
                    if (x < n_classes) c = x;
                }
            }
            key[k] = c;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, c);
        if (k < K && c < n_classes && (peers & lanemask_lt()) == 0) atomicAdd(&dst[c], (unsigned)__popc(peers));
    }
    if (local) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < n_classes; i += blockDim.x)
            if (h[i]) atomicAdd(&cnt[i], h[i]);
    }
}
// Few classes: the kernels grouped by class in one counting pass (kernel order
// kept).  The class is read off the kernel's operator by the count, which keeps
// it for the placing launch (CLASS_DIGIT: none).
constexpr int CLASS_DIGIT = RADIX_BINS - 1;         // and the empty digit that ends the last class
struct ClassDigit {
    const int32_t *rok;
    const uint32_t *r_op, *class_of_op;
    int64_t R, n_ops;
    uint32_t n_classes;
    uint8_t *keep;
    __device__ __forceinline__ unsigned operator()(int64_t k) const {
        unsigned d = CLASS_DIGIT;
        const int32_t r = range_of(rok, r_op, k);
        if (r >= 0 && r < R) {
            const uint32_t op = r_op[r];
            if ((int64_t)op < n_ops) {
                const uint32_t x = class_of_op[op];
                if (x < n_classes) d = x;
            }
        }
        keep[k] = (uint8_t)d;
        return d < CLASS_DIGIT ? d : (unsigned)RADIX_BINS;
    }
};
struct KeptDigit {
    const uint8_t *keep;
    __device__ __forceinline__ unsigned operator()(int64_t k) const {
        const unsigned d = keep[k];
        return d < CLASS_DIGIT ? d : (unsigned)RADIX_BINS;
    }
};
struct PlaceByClass {
    uint32_t *list;
    __device__ __forceinline__ unsigned operator()(int64_t k, uint32_t dest, unsigned) const {
        list[dest] = (uint32_t)k;
        return 0u;
    }
    __device__ __forceinline__ void done(unsigned) const {}
};
// The classes over the warps of the summing pass (one block): class c's kernels
// are list positions [off[c], off[c + 1]); it gets warps [first[c], first[c + 1]),
// in proportion to its kernels and one at least.
__global__ void __launch_bounds__(RADIX_BINS) k_class_warps(const uint32_t *__restrict__ offs, int64_t ntiles,
                                                            int n_classes, uint32_t warps, uint32_t *__restrict__ off,
                                                            uint32_t *__restrict__ first) {
    pdl_wait();
    __shared__ uint32_t wbuf[33];
    const int c = threadIdx.x;
    const uint32_t a = c <= n_classes ? offs[(int64_t)c * ntiles] : 0u;
    const uint32_t z = c < n_classes ? offs[(int64_t)(c + 1) * ntiles] : a;
    const unsigned long long all = offs[(int64_t)n_classes * ntiles];
    const uint32_t share =
        all ? (uint32_t)((unsigned long long)(z - a) * (warps - (uint32_t)n_classes) / all) : 0u;
    const uint32_t ex = block_exclusive_scan<uint32_t>(c < n_classes ? share + 1 : 0u, wbuf, (uint32_t *)nullptr);
    if (c <= n_classes) {
        off[c] = a;
        first[c] = ex;
    }
}
// The classes' sums.  Warp i of a class's m takes every m-th group of 32
// consecutive kernels of its list, so that all warps go through the kernel array
// at one pace and the rows in flight are one band of it: neighbouring rows of
// different classes share their 64-byte pieces of memory, and taken class by
// class each of them was fetched again (220 bytes from memory per kernel).  One
// partial per warp, over a lane's run of kernels / (32 x warps): 105 for 8M kernels on
// 2,432 warps, renormalised like any other.
//
// Bound by issue (some 300 instructions per 32 kernels) and the rows' latency at
// 16 warps per multiprocessor.  8M kernels in 64 classes: class by class in
// pieces of 1,024 318 us, by windows of 32,768 kernels (as many partials as
// windows times classes) 255 us, so 141 us.
__global__ void __launch_bounds__(PC_THREADS, 2) k_class_sums(const uint32_t *__restrict__ off,
                                                              const uint32_t *__restrict__ first, int n_classes,
                                                              const uint32_t *__restrict__ list, AggIn A,
                                                              Acc *__restrict__ part) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char ag_smem[];
    PieceSlots &S = reinterpret_cast<PieceSlots *>(ag_smem)[threadIdx.x / 32];
    const uint32_t g = (blockIdx.x * PC_THREADS + threadIdx.x) >> 5;
    if (g >= first[n_classes]) return;
    int c = 0, hi = n_classes;                    // the warp's class: last one with first <= g
    while (hi - c > 1) {
        const int m = (c + hi) >> 1;
        if (first[m] <= g) c = m; else hi = m;
    }
    const uint32_t m = first[c + 1] - first[c], n = off[c + 1] - off[c], e0 = (g - first[c]) * 32 + lane_id();
    const uint32_t *seg = list + off[c] + e0;
    piece_by_warp(A, [&](uint32_t t) { return seg[(size_t)t * m * 32]; }, e0 < n ? (n - e0 + m * 32 - 1) / (m * 32) : 0u,
                  S, part + g);
}
// One block per class merges its warps' partials: thread t takes t, t +
// FIN_THREADS, ... in order, then the trees of k_agg_long_ops.
__global__ void __launch_bounds__(FIN_THREADS) k_class_records(const uint32_t *__restrict__ first,
                                                               const Acc *__restrict__ part, AggIn A, DevStatus *st) {
    pdl_wait();
    __shared__ Acc wpart[FIN_THREADS / 32];
    const int c = blockIdx.x;
    Acc acc;
    acc.init();
    for (uint32_t p = first[c] + threadIdx.x; p < first[c + 1]; p += FIN_THREADS) acc_merge(acc, part[p]);
#pragma unroll 1
    for (int d = 16; d > 0; d >>= 1) acc_merge_down(acc, d);
    if (lane_id() == 0) wpart[threadIdx.x >> 5] = acc;
    __syncthreads();
    // the last steps weigh most: a thread per counter adds the warps' sums with
    // every rounding carried along, and rounds once (one thread, a pair at a time:
    // 22 us for 64 classes instead of 18, and a third more error)
    __shared__ ff sums[N_SUM + N_DW];
    const int i = threadIdx.x;
    if (i < N_SUM + N_DW) {
        ff x{0.f, 0.f};
        float rest = 0.f;
        for (int v = 0; v < FIN_THREADS / 32; ++v) {
            const ff y = i < N_SUM ? wpart[v].s[i] : wpart[v].w[i - N_SUM];
            const ff t = two_sum(x.hi, y.hi), e = two_sum(x.lo, t.lo), u = two_sum(e.hi, y.lo);
            x = ff{t.hi, u.hi};
            rest = __fadd_rn(rest, __fadd_rn(e.lo, u.lo));
        }
        sums[i] = two_sum(x.hi, __fadd_rn(x.lo, rest));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Acc total = wpart[0];
        for (int v = 1; v < FIN_THREADS / 32; ++v) acc_merge(total, wpart[v]);
#pragma unroll
        for (int q = 0; q < N_SUM; ++q) total.s[q] = sums[q];
#pragma unroll
        for (int q = 0; q < N_DW; ++q) total.w[q] = sums[N_SUM + q];
        total.write(A, c);
        if (total.bad) set_err(st, ERR_INVALID);
    }
}
__global__ void k_iota_u32(uint32_t *dst, int64_t n, unsigned *count) {
    pdl_wait();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = (uint32_t)i;
    if (blockIdx.x == 0 && threadIdx.x == 0) *count = (unsigned)n;
}

opattr_status do_rollup(Ctx &c, const opattr_kernels *kern, const opattr_ranges *rng, const int32_t *rok,
                        const opattr_ncu *ncu, const int32_t *nidx, uint32_t n_ops, const uint32_t *class_of_op,
                        uint32_t n_classes, const opattr_op_aggregates *out) {
    const int64_t K = kern->n, R = rng->n, M = ncu->n, O = n_ops, C = n_classes;
    if (K < 0 || R < 0 || M < 0 || K >= (1ll << 31) || R >= (1ll << 31) || M >= (1ll << 31) || !out)
        return OPATTR_E_INVALID_ARG;
    if (C > (1 << 24)) return OPATTR_E_INVALID_ARG;
    if (K > 0 && (!kern->dur_ns || !nidx)) return OPATTR_E_INVALID_ARG;
    if (K > 0 && !rok && R != K) return OPATTR_E_INVALID_ARG;
    if (R > 0 && !rng->op_id) return OPATTR_E_INVALID_ARG;
    if (O > 0 && !class_of_op) return OPATTR_E_INVALID_ARG;
    if (M > 0 && !ncu->counters) return OPATTR_E_INVALID_ARG;
    if (C > 0 && (!out->kernel_count || !out->total_duration_ns || !out->matched_count || !out->agg))
        return OPATTR_E_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(ncu->counters) & 15) != 0) return OPATTR_E_INVALID_ARG;

    // few classes: one counting pass, every warp of one wave for a share of one
    // class; else a sort by class and pieces
    const bool few = K > 0 && C > 0 && C <= CLASS_DIGIT;
    const int sms = sm_count(c);
    const unsigned sum_blocks = (unsigned)std::min<int64_t>(2 * sms, (K + 32 * 64 - 1) / (32 * 64) + C / 8 + 1);
    const uint32_t sum_warps = sum_blocks * (PC_THREADS / 32);
    const int64_t maxp = std::max<int64_t>(K / AG_PIECE + C + 1, sum_warps);
    Need nd;
    for (int i = 0; i < 4; ++i) nd.add<uint32_t>(K);
    nd.add<uint32_t>(radix_hist_elems(K)).add<uint32_t>(scan_scratch_elems(std::max(radix_hist_elems(K), C + 2)));
    nd.add<uint32_t>(C + 2).add<uint32_t>(C + 2).add<uint32_t>(C + 1).add<uint32_t>(C + 1).add<unsigned>(1);
    nd.add<Acc>(maxp);
    opattr_status st = ensure_arena(c, nd.bytes + 4096);
    if (st) return st;
    Arena a(c);
    if ((st = reset_status(c))) return st;
    uint32_t *k0 = a.take<uint32_t>(K), *v0 = a.take<uint32_t>(K), *k1 = a.take<uint32_t>(K), *v1 = a.take<uint32_t>(K);
    uint32_t *hist = a.take<uint32_t>(radix_hist_elems(K));
    uint32_t *part = a.take<uint32_t>(scan_scratch_elems(std::max(radix_hist_elems(K), C + 2)));
    uint32_t *cnt = a.take<uint32_t>(C + 2), *off = a.take<uint32_t>(C + 2);
    uint32_t *cls = a.take<uint32_t>(C + 1), *poff = a.take<uint32_t>(C + 1);
    unsigned *ncls = a.take<unsigned>(1);
    Acc *partials = a.take<Acc>(maxp);
    if (!k0 || !v0 || !k1 || !v1 || !hist || !part || !cnt || !off || !cls || !poff || !ncls || !partials)
        return OPATTR_E_OOM;
    if (O > 0)
        launch(c, "class_check", k_class_check, dim3(grid_for(O, 256, REDUCE_GRID)), dim3(256), 0, class_of_op, O,
               n_classes, c.d_status);
    uint32_t *list = nullptr;
    if (few) {
        uint8_t *keep = reinterpret_cast<uint8_t *>(v0);
        const ClassDigit dg{rok, rng->op_id, class_of_op, R, O, n_classes, keep};
        list = k0;
        const uint32_t *offs = digit_offsets(c, dg, K, hist, part, (int)C + 1);
        digit_rank(c, "class_place", KeptDigit{keep}, K, offs, PlaceByClass{list});
        launch(c, "class_warps", k_class_warps, dim3(1), dim3(RADIX_BINS), 0, offs, (K + RADIX_TILE - 1) / RADIX_TILE,
               (int)C, sum_warps, off, poff);
    } else {
        const ZeroRun z{cnt, C + 2};
        if ((st = zero_runs(c, 1, &z))) return st;
    }
    if (K > 0 && !few) {
        launch(c, "class_keys", k_class_keys, dim3(grid_for(K, 256, REDUCE_GRID)), dim3(256), 0, rok, rng->op_id, K, R,
               O, class_of_op, n_classes, k0, cnt);
        uint32_t *ko;
        radix_sort_pairs<uint32_t>(c, k0, v0, k1, v1, K, bits_for((uint64_t)C), true, hist, part, &ko, &list);
    }
    if (!few) scan_exclusive_u32(c, cnt, off, C + 1, part, nullptr);   // off[C] = kernels with a class
    if (C > 0) {
        AggIn in{};
        in.dur = kern->dur_ns;
        in.ncu_idx = nidx;
        in.counters = ncu->counters;
        in.M = M;
        in.n_ops = C;
        in.lane_max = 0;
        in.ctr = nullptr;
        in.dirty = nullptr;
        in.mids = nullptr;
        in.longs = nullptr;
        in.nonident = nullptr;
        in.out = *out;
        if (few) {
            cudaFuncSetAttribute(k_class_sums, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PC_SMEM);
            launch(c, "class_sums", k_class_sums, dim3(sum_blocks), dim3(PC_THREADS), PC_SMEM, (const uint32_t *)off,
                   (const uint32_t *)poff, (int)C, (const uint32_t *)list, in, partials);
            launch(c, "class_records", k_class_records, dim3((unsigned)C), dim3(FIN_THREADS), 0,
                   (const uint32_t *)poff, (const Acc *)partials, in, c.d_status);
        } else {
            launch(c, "class_iota", k_iota_u32, dim3(grid_for(C, 256, 4096)), dim3(256), 0, cls, C, ncls);
            launch(c, "agg_piece_offsets", k_agg_piece_offsets, dim3(1), dim3(1024), 0, (const uint32_t *)off,
                   (const uint32_t *)cls, (const unsigned *)ncls, poff);
            if (K > 0) launch_pieces(c, off, list, cls, ncls, poff, in, partials);
            launch(c, "class_records", k_agg_long_ops, dim3(2 * sms), dim3(FIN_THREADS), 0, (const uint32_t *)cls,
                   (const unsigned *)ncls, (const uint32_t *)poff, (const Acc *)partials, in, c.d_status);
        }
    }
    if ((st = read_status(c))) return st;
    if (c.h_status->err & ERR_INVALID) return OPATTR_E_INVALID_ARG;
    return OPATTR_OK;
}

}  // namespace opattr
