// common.cuh -- context, scratch arena, launch accounting and device helpers
// shared by the kernels of libopattr.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <string>
#include <vector>

#include "opattr.h"

namespace opattr {

// ------------------------------------------------------------------ status block
// One small struct in device memory per context, reset at the start of each
// call and read back at its checkpoints.  Kernels never trap: they record
// problems here and return.
enum ErrBit : unsigned {
    ERR_INVALID = 1u,     // bad id, value or size found on the device
    ERR_NOT_NESTED = 2u,  // ranges are not laminar
    ERR_DEPTH = 4u,       // depth > 31
    ERR_TIMEOUT = 8u,     // a bounded wait gave up
    ERR_COUNT = 16u,      // count mismatch in error mode
};
enum FlagBit : unsigned {
    F_K_UNSORTED = 1u,    // kernels are not in (start, stream) order
    F_R_UNSORTED = 2u,    // ranges are not in start order
    F_LEVEL_FIXUP = 4u,   // equal starts in a level are not in end order
    F_NAMES_DIFFER = 8u,  // ncu names differ from replayed names in time order
    F_OP_DUP = 16u,       // two operator ranges share an op id
    F_AGG_MISS = 32u,     // the owned-range aggregation missed kernels
    F_IDX_NOT_ID = 64u,   // some kernel's ncu row index is neither its own index nor -1
    F_LEVELS_MANY = 128u, // more range levels than the enclosure's common layout holds
    F_TIMES_FAR = 256u,   // events too far apart for the enclosure's 32-bit times
    // the enclosure has to run again
    F_REDO = F_K_UNSORTED | F_R_UNSORTED | F_LEVEL_FIXUP | F_LEVELS_MANY | F_TIMES_FAR,
};
enum CountSlot {
    C_NAMES_MISMATCH = 0,
    C_COUNT_UNMATCHED,
    C_DIRECT,
    C_BROADCAST,
    C_DEDUP_MISMATCH,
    C_REPLAYED,
    C_TOTAL_NS,
    C_ATTR_NS,
    C_ATTR_K,
    C_MATCHED_K,
    C_AGG_SEEN,
    C_UNMATCHED,
    C_TIER_HIGH,
    C_TIER_NVTX,
    C_TIER_INDUCTOR,
    C_FUSED,
    C_CORR_USED,
    C_MAX_KEY,               // largest matching key of kernels and rows
    C_NSLOTS = 24
};
enum MinMaxSlot { MM_KSTART_MIN = 0, MM_KSTART_MAX, MM_RSTART_MIN, MM_REND_MAX, MM_NSLOTS = 8 };

struct DevStatus {
    unsigned int err;
    unsigned int flags;
    unsigned long long cnt[C_NSLOTS];
    long long mm[MM_NSLOTS];
    unsigned int kstreams[8];    // streams with kernels, one bit each (the enclosure's checks)
};

// ------------------------------------------------------------------ context
struct TimingSlot {
    const char *name;
    double total_ms;
    int64_t launches;
};

constexpr int N_LEVELS = 256 * 32;   // (stream, depth) levels of the enclosure
constexpr size_t STAGE_BYTES = 32768;  // pinned staging of host-built tables
constexpr int SMALL_WORDS = 512;

struct Ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int sms = 0;                     // multiprocessors of the device (sm_count)
    cudaEvent_t ev_status = nullptr; // a status copy under way (post_status); created on first use
    opattr_config cfg{};
    bool broken = false;
    // scratch arena (bump allocation, reset per call)
    char *arena = nullptr;
    size_t arena_cap = 0, arena_used = 0;
    bool arena_fixed = false;        // the arena is caller-provided memory: never grow or free it
    // status block
    DevStatus *d_status = nullptr;
    DevStatus *h_status = nullptr;   // pinned mirror
    uint32_t *h_small = nullptr;     // pinned room for a few values read mid-call [SMALL_WORDS]
    unsigned char *h_stage = nullptr; // pinned staging for small host-built tables [STAGE_BYTES]
    bool host_mapped = false;        // the three pinned buffers above are addressable from the device as they are
    // kernel time order as the last enclosure found it (-1 unknown, 0 / 1),
    // and whether the matching may take it instead of checking again (join)
    int enclose_k_sorted = -1;
    bool order_from_enclose = false;
    // within a join: the enclosure's kernel time order (unsorted kernels), kept
    // for the matching at the start of the arena (arena_keep bytes survive the
    // per-call resets and any growth of the arena)
    bool in_join = false;
    uint32_t *join_korder = nullptr;
    size_t arena_keep = 0;
    // within a join: the matching's identity pairing (rows equal to the
    // kernels in time order), done by the enclosure's checking pass when
    // spec_k > 0; spec_ran: it was, its verdict in the status the enclosure
    // read last
    const uint32_t *spec_kname = nullptr, *spec_nname = nullptr;
    int32_t *spec_idx = nullptr;
    uint8_t *spec_kind = nullptr;
    int64_t spec_k = 0;
    bool spec_ran = false;
    // within a join whose matching must sort its names: the largest key, found
    // by the enclosure's checking pass (max_ncu), then max_known
    const opattr_ncu *max_ncu = nullptr;
    bool max_known = false;
    // within a join: the matching's results are complete but its counts and
    // verdict are read with the aggregation's status (match_pending); then the
    // aggregation keeps the status block (keep_status).  no_spec: the fast
    // pairing is known to fail
    bool match_pending = false, keep_status = false, no_spec = false;
    opattr_match_summary match_sum{};
    // within a join whose matching can be skipped: the enclosure's last status
    // read is left to the aggregation's (defer_status), and the enclosure's
    // verdict is pending until then (enclose_pending; the aggregation keeps
    // the status block instead of resetting it)
    bool defer_status = false, enclose_pending = false;
    unsigned redo = 0;               // why the enclosure's deferred run did not do (F_REDO bits)
    // within a join: the matching was the identity pairing (row k for kernel
    // k), so the aggregation need not read the row indices
    bool rows_identity = false;
    // within a join: the aggregation's counters, agg_words of them at the start
    // of the arena, are zeroed by the enclosure's reset (agg_ready) unless the
    // arena has to grow on the way
    int64_t agg_words = 0;
    bool agg_ready = false;
    // within a join: scratch that its matching and aggregation will ask for on
    // records in order (beyond what is kept), so that the enclosure's request is
    // the join's only one
    size_t join_scratch = 0;
    // launch accounting
    int64_t launches = 0;
    bool timing = false;
    std::string timing_only;         // with timing on: bracket only this kernel (empty = all)
    std::vector<TimingSlot> slots;
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> pending;
    std::vector<cudaEvent_t> event_pool;
    cudaError_t last_error = cudaSuccess;
};

// ------------------------------------------------------------------ scratch
struct Arena {
    Ctx &c;
    explicit Arena(Ctx &ctx) : c(ctx) { c.arena_used = c.arena_keep; }
    template <typename T>
    T *take(int64_t count) {
        size_t bytes = (size_t)(count > 0 ? count : 1) * sizeof(T);
        size_t at = (c.arena_used + 255) & ~(size_t)255;
        if (at + bytes > c.arena_cap) return nullptr;
        c.arena_used = at + bytes;
        return reinterpret_cast<T *>(c.arena + at);
    }
};
// Upper bound of an arena request made of several arrays (alignment slack included).
struct Need {
    size_t bytes = 0;
    template <typename T>
    Need &add(int64_t count) {
        bytes += (((size_t)(count > 0 ? count : 1) * sizeof(T)) + 255) & ~(size_t)255;
        return *this;
    }
};

opattr_status ensure_arena(Ctx &c, size_t bytes);
int sm_count(Ctx &c);
// The status of an enclosure that read `H` (a NOT_NESTED found beside
// F_LEVEL_FIXUP does not count: the run on sorted ranges decides).
opattr_status enclose_verdict(const DevStatus &H, int64_t K);
// Words of the aggregation's counters for n_ops operators: a few of its own,
// the status words of the scan, and one per operator and one more.
constexpr int AGG_OWN_WORDS = 8;
int64_t agg_counter_words(uint32_t n_ops);
// Scratch (bytes) of the aggregation beside those counters, and of the matching.
size_t aggregate_scratch(int64_t K, uint32_t n_ops);
size_t match_scratch(int64_t K, int64_t M, bool dedup_on, int64_t n_layers);
// The matching's counts and status from the status block (c.match_sum holds
// what was known before it ran).
opattr_status match_verdict(Ctx &c, opattr_match_summary *sum);
// A small transfer between the context's pinned host buffers and device
// memory, on c.stream.  When those buffers are mapped into the device's
// address space (opattr_create checks), a small kernel moves the bytes through
// the mapping instead of a copy engine, so a call's status reads and table
// uploads never queue behind bulk copies that the caller has on the engines;
// otherwise (host mirrors in plain host memory) cudaMemcpyAsync.
opattr_status copy_small(Ctx &c, void *dst, const void *src, size_t bytes, cudaMemcpyKind kind);
struct SmallCopy {
    void *dst;
    const void *src;
    size_t bytes;
};
// Several such transfers of one direction, four to a launch.
opattr_status copy_small_n(Ctx &c, int count, const SmallCopy *cp, cudaMemcpyKind kind);
// Words to be zeroed, up to four runs in one launch; with reset_status in the
// launch that resets the status block.
struct ZeroRun {
    void *p;
    int64_t words;
};
opattr_status zero_runs(Ctx &c, int n, const ZeroRun *z);
opattr_status reset_status(Ctx &c, int n = 0, const ZeroRun *z = nullptr);
// The status block sent to the host without waiting (with up to three more
// transfers in the launch), and the wait for it alone: work queued after
// post_status goes on meanwhile.
opattr_status post_status(Ctx &c, int n_extra = 0, const SmallCopy *extra = nullptr);
opattr_status await_status(Ctx &c);
// The status block back to the host (with up to three more device->host
// transfers in the same launch), then a stream synchronize.
opattr_status read_status(Ctx &c, int n_extra = 0, const SmallCopy *extra = nullptr);
// The same where a kernel on the stream has stored the block to h_status itself.
opattr_status sync_status(Ctx &c);
opattr_status cuda_status(Ctx &c, cudaError_t e);
int timing_slot(Ctx &c, const char *name);
void timing_begin(Ctx &c, int slot, cudaEvent_t *e0, cudaEvent_t *e1);
void timing_end(Ctx &c, int slot, cudaEvent_t e0, cudaEvent_t e1);
void timing_collect(Ctx &c);             // after a stream synchronize

// Launch a kernel on the context stream, counting it and (optionally) timing
// it.  Kernels go out as programmatic dependent launches: the next kernel of
// the stream is set up and its blocks scheduled while this one's last blocks
// finish, instead of after its completion; every kernel of the library calls
// pdl_wait() before its first memory access, which holds it until the
// kernel before it has completed and its writes are visible.
template <typename... KArgs, typename... Args>
inline void launch(Ctx &c, const char *name, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                   Args... args) {
    if (grid.x == 0 || grid.y == 0 || grid.z == 0) return;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int slot = -1;
    const bool timed = c.timing && (c.timing_only.empty() || c.timing_only == name);
    if (timed) {
        slot = timing_slot(c, name);
        timing_begin(c, slot, &e0, &e1);
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c.stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, args...);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess && c.last_error == cudaSuccess) c.last_error = e;
    c.launches++;
    if (timed) timing_end(c, slot, e0, e1);
}

inline unsigned grid_for(int64_t n, int per_block, unsigned cap = 1u << 30) {
    int64_t g = (n + per_block - 1) / per_block;
    if (g < 1) g = 1;
    return (unsigned)(g > (int64_t)cap ? cap : g);
}

// ------------------------------------------------------------------ device helpers
// The first statement of every kernel: waits, under a programmatic dependent
// launch, until the kernel before it in the stream has completed and its
// memory is visible (returns at once otherwise).  No kernel signals early
// completion, so a kernel's blocks never hold resources that the blocks of
// the kernel before it still need.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Lanes of the warp whose 8-bit digit equals this lane's, among the lanes
// with `valid` set: one ballot per digit bit (the rank-by-digit step of a
// stable multi-split).
__device__ __forceinline__ unsigned warp_peers8(unsigned d, bool valid) {
    unsigned m = __ballot_sync(0xffffffffu, valid);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        const bool bit = (d >> b) & 1u;
        const unsigned x = __ballot_sync(0xffffffffu, bit);
        m &= bit ? x : ~x;
    }
    return m;
}

__device__ __forceinline__ void set_err(DevStatus *s, unsigned bit) { atomicOr(&s->err, bit); }
__device__ __forceinline__ void set_flag(DevStatus *s, unsigned bit) { atomicOr(&s->flags, bit); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if ((int)lane_id() >= o) v += u;
    }
    return v;
}

// Exclusive scan over a block (blockDim.x a multiple of 32, <= 1024).
// `warp_buf` holds 33 entries of shared memory.  Returns the exclusive prefix;
// *total receives the block sum.
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *warp_buf, T *total) {
    const unsigned w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = warp_inclusive_scan(v);
    if (lane_id() == 31) warp_buf[w] = inc;
    __syncthreads();
    if (w == 0) {
        T x = lane_id() < nw ? warp_buf[lane_id()] : T(0);
        T xs = warp_inclusive_scan(x);
        if (lane_id() < nw) warp_buf[lane_id()] = xs - x;
        if (lane_id() == nw - 1) warp_buf[32] = xs;
    }
    __syncthreads();
    T r = warp_buf[w] + inc - v;
    if (total) *total = warp_buf[32];
    __syncthreads();
    return r;
}

template <typename T>
__device__ __forceinline__ T block_sum(T v, T *warp_buf) {
    T total;
    block_exclusive_scan(v, warp_buf, &total);
    return total;
}

// p[0 .. n) = 0 by the whole grid: scratch of the launch after this one.
__device__ __forceinline__ void zero_words(uint32_t *p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = 0;
}

// Sum v over the block and add the total to *dst with one atomic.  Every
// thread of the block must call it (it synchronises the block).
__device__ __forceinline__ void block_add_u64(unsigned long long v, unsigned long long *dst,
                                              unsigned long long *warp_buf) {
    unsigned long long t = block_sum<unsigned long long>(v, warp_buf);
    if (threadIdx.x == 0 && t) atomicAdd(dst, t);
}

// Blocks for grid-stride reductions: enough to fill the GPU, few enough that
// one atomic per block stays cheap.
constexpr unsigned REDUCE_GRID = 2048;

}  // namespace opattr
