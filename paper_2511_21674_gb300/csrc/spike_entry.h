// A spike in the list of the batched single-window gradient: its row of the
// window tables, relative to a base, and the steps of the window after it.
// Plain integer functions, shared with host code.
#pragma once
#include <stdint.h>

#ifndef EPROP_HD
#ifdef __CUDACC__
#define EPROP_HD __host__ __device__ __forceinline__
#else
#define EPROP_HD inline
#endif
#endif

namespace eprop {

// The tables hold one row per (sample, arrival step 1..U), sample after
// sample: arrival a of sample b is row b U + a - 1.  A spike word holds 32
// steps of one sample, so the rows of the words w0 .. w0 + kEntrySpan - 1 stay
// below 32 kEntrySpan above the first word's first row: 28 bits.  The upper
// four bits hold the steps after the spike, clipped (delays are at most 8).
// (Sample and step side by side in 32 bits bounded both: 2^11 and 2^20.)
constexpr int kEntryRowBits = 28;
constexpr int kEntrySpan = 1 << (kEntryRowBits - 5);       // words one base serves
constexpr int kEntryMaxAfter = 15;

// table row one before the arrivals of a spike at bit 0 of word k of sample b
EPROP_HD long long entry_base(int b, int k, int U) { return (long long)b * U + (long long)k * 32 - 1; }

EPROP_HD uint32_t entry_pack(long long base, int b, int step, int U, int T) {
    const int after = T - step < kEntryMaxAfter ? T - step : kEntryMaxAfter;
    return (uint32_t)((long long)b * U + step - 1 - base) | ((uint32_t)after << kEntryRowBits);
}

// whether the spike's arrival d steps later lies inside the window, and its row
EPROP_HD bool entry_arrives(uint32_t e, int d) { return d <= (int)(e >> kEntryRowBits); }
EPROP_HD long long entry_row(long long base, uint32_t e, int d) {
    return base + (long long)(e & ((1u << kEntryRowBits) - 1u)) + d;
}

}  // namespace eprop
