// util.cuh -- steps shared by the three calls: kernel time-order check and
// time-order permutation.
#pragma once
#include "common.cuh"
#include "sort.cuh"

namespace opattr {

// Sets F_K_UNSORTED unless (start_ns, stream) is non-decreasing along the
// array, and records min / max start in MM_KSTART_MIN / MM_KSTART_MAX.
void check_kernel_order(Ctx &c, const uint8_t *stream, const int64_t *start, int64_t n);

// Scratch (bytes) of a time sort of n records (kernel_time_order).
size_t time_sort_scratch(int64_t n);

// Permutation of kernel indices into time order (start, stream, index): sorted
// by (start - min_start) << sbits | stream.  Needs the min / max from
// check_kernel_order (or the enclosure's checks) in c.h_status.  With scmap (device, [256]: increasing
// compact ids of the streams that have kernels) the key holds the compact id
// in stream_bits bits instead of the id in 8.  *order receives a device array
// of n indices carved from `a`, *keys (if given) the sorted keys
// (OPATTR_E_INVALID_ARG where they would not fit 64 bits).  May wait on the stream
// (and reads the status block then).
opattr_status kernel_time_order(Ctx &c, struct Arena &a, const uint8_t *stream, const int64_t *start, int64_t n,
                                uint32_t **order, const uint8_t *scmap = nullptr, int stream_bits = 8,
                                uint64_t **keys = nullptr);

// The same for ranges: sorted by (start - tmin) << 6 | depth << 1 | (longer than
// zero), with tmin the smallest start and tmax no smaller than the largest; *keys
// is NULL where tmax - tmin leaves no room for the six bits.
constexpr int RANGE_KEY_SHIFT = 6;
opattr_status range_time_order(Ctx &c, struct Arena &a, const int64_t *start, const int64_t *end,
                               const uint8_t *depth, int64_t n, long long tmin, long long tmax, uint32_t **order,
                               uint64_t **keys);

}  // namespace opattr
