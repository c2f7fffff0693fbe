// Counting by partial patterns (partial.cu): the arguments of its kernels.
#pragma once

#include <vector>

#include "common.cuh"

namespace acc {

// Counts by state in one word: three fields of kNdBits bits, state 1 lowest
// (typed degrees; typed common neighbours of an edge, a word per state to the
// one end).  No count exceeds a degree, and degrees are at most kNdMax.
constexpr int kNdBits = 21;
constexpr int kNdMax = (1 << kNdBits) - 1;

struct PartialArgs {
    const uint32_t *state;      // the graph set, as EnumArgs
    uint32_t *state_w;          // the same pair-state buffer, to clear
    const int *deg, *lo;
    const long long *nptr;
    const uint32_t *nbr, *src;
    const uint32_t *nh;         // hashed adjacency, or NULL: probes read the dense block
    const int16_t *lut;         // class table in the state-vector layout
    const uint32_t *inv;        // partial_matrix
    GSet gs;
    GraphInfo *info;
    uint4 *queue;               // k = 4: ranges of heavy roots (vertex, first and last end, graph)
    unsigned long long queue_cap;
    uint2 *rev;                 // k = 4: reverse positions of the upper entries
    unsigned long long *nd;     // typed degrees by global vertex (zeroed by the caller)
    uint32_t *wedges;           // k = 4: wedges of each root (zeroed by the caller)
    unsigned long long *tri;    // k = 4: three words per neighbour entry
    unsigned long long *part;   // partial counts, B * num_classes (zeroed by the caller)
    int *done;                  // finished slices per graph (zeroed by the caller)
    int slices;
    unsigned long long *counts; // B * num_classes
    int *status;
    const uint32_t *occ;        // occupancy bitmap of the dense block to clear, or NULL
    int occ_w;
};

// The matrix from partial counts to induced ones (k = 3, 4): the number of its
// entries, then (to << 24) | (from << 16) | (coefficient + 2^15).  lut,
// class_code: the class table in the canonical layout (host).
void partial_matrix(int k, const int16_t *lut, const uint32_t *class_code, std::vector<uint32_t> &out);

// Counts the built set (k = 3, 4; largest degree at most kNdMax) and clears
// its dense block; max_entries bounds 2 |E*|.  Returns the launches.
int launch_partial(int k, PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s, int grid_num = 1,
                   int grid_den = 1);

}  // namespace acc
