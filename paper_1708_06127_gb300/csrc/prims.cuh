// Device-wide primitives (scan, radix sort) written for this library; no CUB.
#pragma once
#include "common.cuh"

namespace vc {

// Exclusive prefix sum out[i] = sum_{j<i} in[i]; *total (device pointer, may be
// null) receives the sum of all n inputs; out2 and total2 (may be null) a second copy of
// each.  scratch must hold scan_scratch_elems(n) values of Out.
template <typename In, typename Out>
void exclusive_scan(const In* in, Out* out, int64_t n, Out* total, Out* scratch, cudaStream_t s, Out* out2 = nullptr,
                    Out* total2 = nullptr);
int64_t scan_scratch_elems(int64_t n);

// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the keys.
// The alt buffers are of the same size; the sorted output lands in one pair of buffers or
// the other, and keys/vals point at it afterwards (keys_alt/vals_alt at the rest).
// hist must hold radix_hist_elems(n) int64 values.
void radix_sort_pairs(unsigned long long*& keys, long long*& vals, unsigned long long*& keys_alt,
                      long long*& vals_alt, int64_t n, int bits, long long* hist, cudaStream_t s);
int64_t radix_hist_elems(int64_t n);

}  // namespace vc
