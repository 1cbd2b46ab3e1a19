// Split of a step's delivery into work items: every spiking row in
// 2^delivery_part_shift parts, a hub row in parts of kHubPart records.  Plain
// integer functions, shared with host code.
#pragma once
#include <algorithm>
#include <vector>

#ifndef EPROP_HD
#ifdef __CUDACC__
#define EPROP_HD __host__ __device__ __forceinline__
#else
#define EPROP_HD inline
#endif
#endif

namespace eprop {

// Four parts per row, more where rows are long: at least 512 records per part
// of a row of average length.  Quarter rows of 10,000 synapses kept 2.1 blocks
// busy per SM on average but three on some, and those set the time (scaling
// network 84.8 -> 72 ms per call); at 1000 synapses per row 4 parts measured
// best.  The average, not the longest row: one input onto all of 3e5 neurons
// would cut the others' rows of 100 into 512 items, each with its own look-ups
// and copies (100 steps with 5 input spikes 319 ms; now 19.4 ms).
inline int delivery_part_shift(long long nnz, long long n_src) {
    const long long mean = n_src > 0 ? nnz / n_src : 0;
    int ps = 2;
    while ((mean >> (ps + 1)) >= 512 && ps < 10) ++ps;
    return ps;
}

// Rows far longer than the average (inputs onto every neuron) in parts of their
// own, or their few parts set the time of a step.  Hub rows are those whose part
// would exceed kHubPart records; at most kMaxHubs of them, the longest (one
// thread of a block each looks whether it spiked).  64,000 neurons with rows of
// 1000, 50 inputs onto all of them, 500 steps: 15.0 ms without, 10.5 with.
constexpr int kHubPart = 1024;
constexpr int kMaxHubs = 256;

struct HubRows {
    long long len;               // rows longer than this are hubs
    int n, parts;                // rows listed, parts of the longest one
    int src[kMaxHubs];
};

// the length that hub rows exceed
inline long long delivery_hub_length(const long long *row_ptr, long long n_src, int part_shift) {
    const long long floor = (long long)kHubPart << part_shift;
    std::vector<long long> len;
    for (long long i = 0; i < n_src; ++i)
        if (row_ptr[i + 1] - row_ptr[i] > floor) len.push_back(row_ptr[i + 1] - row_ptr[i]);
    if (len.size() <= (size_t)kMaxHubs) return floor;
    std::nth_element(len.begin(), len.begin() + kMaxHubs, len.end(), [](long long a, long long b) { return a > b; });
    return len[kMaxHubs];
}

// items of `rows` spiking rows (more than 2^31 from 2^21 rows of 2^10 parts on)
EPROP_HD long long delivery_items(int rows, int part_shift) { return (long long)rows << part_shift; }

// records [begin, end) of part `part` of a row of len records
EPROP_HD long long delivery_part_begin(long long len, int part, int part_shift) { return (len * part) >> part_shift; }

}  // namespace eprop
