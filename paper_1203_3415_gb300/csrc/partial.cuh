// Counting by partial patterns: the arguments of its kernels (partial.cu,
// partial5.cu) and their common device functions.
#pragma once

#include <vector>

#include "common.cuh"

namespace acc {

// Counts by state in one word: three fields of kNdBits bits, state 1 lowest
// (typed degrees; typed common neighbours of an edge, a word per state to the
// one end).  No count exceeds a degree, and degrees are at most kNdMax.
constexpr int kNdBits = 21;
constexpr int kNdMax = (1 << kNdBits) - 1;

// k = 5: most neighbours above a root (rows of its pass); the 5-cycle tables count
// a root's wedges to one end in 10 bits, and no more of them than its rows.
constexpr int kCycleRows = 1023;

// k = 5: what the passes share besides the graph (one graph, not a set).
struct Partial5 {
    // counters, zeroed by the caller: triangles listed; set when the set must
    // be counted by the list scan (enum.cu) instead; then unit and queue
    // counters of the pair and the 5-cycle pass
    unsigned long long *ctr;
    uint4 *tris;                // triangles v < u < w: positions of v -> u, u -> w, v -> w
    unsigned long long tri_cap;
    int *in_tri;                // by vertex: nonzero when in a triangle (zeroed by the caller)
    uint32_t *pair_wedges;      // by root v: wedges v - b - w, w above v, any b (zeroed by the caller)
    uint32_t *cycle_wedges;     // by root: its wedges, as PartialArgs::wedges (zeroed by the caller)
    unsigned long long *sums;   // by class: accumulated sums (zeroed by the caller)
    unsigned long long *small;  // classes of k = 3, then arcs by state 1 and 3 (zeroed by the caller)
    const int16_t *lut5, *lut5_canon, *lut4_canon, *lut3, *lut3_canon;
    const uint32_t *code5;      // canonical code by class
    const unsigned char *div5;  // divisor of each class's sum
    const unsigned char *aut3, *aut4;  // automorphisms by class
};
enum { kCtrTris = 0, kCtrScan = 1, kCtrPairUnit, kCtrPairTail, kCtrPairHead, kCtrCycUnit, kCtrCycTail, kCtrCycHead,
       kCtrDiamond, kCtrUnit4, kCtrTail4, kCtrHead4, kCtrs };

struct PartialArgs {
    const uint32_t *state;      // the graph set, as EnumArgs
    uint32_t *state_w;          // the same pair-state buffer, to clear
    const int *deg, *lo;
    const long long *nptr;
    const uint32_t *nbr, *src;
    const uint32_t *nh;         // hashed adjacency, or NULL: probes read the dense block
    const int16_t *lut;         // class table in the state-vector layout (k = 5: of k = 4)
    const uint32_t *inv;        // partial_matrix
    GSet gs;
    GraphInfo *info;
    uint4 *queue;               // parts of the roots with many wedges
    unsigned long long queue_cap;
    uint2 *rev;                 // k = 4: reverse positions of the upper entries; k = 5: of all
    unsigned long long *nd;     // typed degrees by global vertex (zeroed by the caller)
    uint32_t *wedges;           // k = 4, 5: wedges of each root (zeroed by the caller)
    unsigned long long *tri;    // k = 4, 5: three words per neighbour entry
    unsigned long long *part;   // partial counts, B * num_classes (k = 5: of k = 4; zeroed by the caller)
    int *done;                  // finished slices per graph (zeroed by the caller)
    int slices;
    unsigned long long *counts; // B * num_classes
    int *status;
    const uint32_t *occ;        // occupancy bitmap of the dense block to clear, or NULL
    int occ_w;
    Partial5 p5;
};

__device__ __forceinline__ uint32_t swap_state(uint32_t s) { return ((s & 1u) << 1) | (s >> 1); }

// One graph's arrays by local vertex (neighbour-list positions are global).
struct PView {
    const uint32_t *state;
    long long pitch;
    const long long *nptr;
    const int *deg, *lo;
    const unsigned long long *nd;
    const uint32_t *nh;
    int n;
};

__device__ __forceinline__ PView pview(const PartialArgs &a, const GMeta &mt) {
    return PView{a.state + mt.soff, mt.pitch,        a.nptr + mt.voff, a.deg + mt.voff,
                 a.lo + mt.voff,    a.nd + mt.voff, a.nh,             mt.n};
}

// state(x, y): the dense block, or x's hashed table (enum.cu, nh.cu).
template <bool HASH>
__device__ __forceinline__ uint32_t pstate(const PView &g, uint32_t x, uint32_t y) {
    if constexpr (HASH) {
        const uint32_t lg = nh_lg(g.deg[x]), m = (1u << lg) - 1u;
        const uint4 *tab = reinterpret_cast<const uint4 *>(g.nh + (long long)kNhWords * g.nptr[x]);
        uint32_t k = nh_bucket(y, lg);
        for (uint32_t tries = 0; tries <= m; tries++, k = (k + 1u) & m) {
            const uint4 q = __ldg(tab + k);
            if ((q.x >> 2) == y) return q.x & 3u;
            if ((q.y >> 2) == y) return q.y & 3u;
            if ((q.z >> 2) == y) return q.z & 3u;
            if ((q.w >> 2) == y) return q.w & 3u;
            if (!q.w) return 0u;
        }
        return 0u;
    } else {
        return (__ldg(g.state + (long long)x * g.pitch + (y >> 4)) >> ((y & 15u) << 1)) & 3u;
    }
}

// First index of the sorted entries e[0..n) (u << 2 | state) with u >= id.
__device__ __forceinline__ int lower_id(const uint32_t *__restrict__ e, int n, uint32_t id) {
    const uint32_t key = id << 2;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(e + mid) < key) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// The part of the sorted entries e[*first .. *first + n) with ids in [lo, hi):
// its length, *first moved to its start (both ends searched side by side: the
// loads of one wait beside the other's).
__device__ __forceinline__ int id_range(const uint32_t *__restrict__ e, int n, uint32_t lo, uint32_t hi,
                                        uint32_t *first) {
    const uint32_t *__restrict__ x = e + *first;
    const uint32_t k0 = lo << 2, k1 = hi << 2;
    int a0 = 0, b0 = n, a1 = 0, b1 = n;
    while (a0 < b0 || a1 < b1) {
        const int m0 = (a0 + b0) >> 1, m1 = (a1 + b1) >> 1;
        const uint32_t y0 = a0 < b0 ? __ldg(x + m0) : 0u, y1 = a1 < b1 ? __ldg(x + m1) : 0u;
        if (a0 < b0) {
            if (y0 < k0) a0 = m0 + 1;
            else b0 = m0;
        }
        if (a1 < b1) {
            if (y1 < k1) a1 = m1 + 1;
            else b1 = m1;
        }
    }
    *first += (uint32_t)a0;
    return a1 - a0;
}

__device__ __forceinline__ int warp_excl(int x, int lane, int *total) {
    int incl = x;
#pragma unroll
    for (int d = 1; d < kWarp; d <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += y;
    }
    *total = __shfl_sync(kFull, incl, kWarp - 1);
    return incl - x;
}

// 64-bit histogram bin in shared memory as two words (the hardware adds 32
// bits natively): the add that carries out of the low word raises the high.
__device__ __forceinline__ void hist_add(uint32_t *h, int bin, unsigned long long d) {
    const uint32_t lo = (uint32_t)d;
    uint32_t hi = (uint32_t)(d >> 32);
    if (lo) {
        const uint32_t old = atomicAdd(&h[2 * bin], lo);
        if (old > ~lo) hi++;
    }
    if (hi) atomicAdd(&h[2 * bin + 1], hi);
}

__device__ __forceinline__ unsigned long long nd_of(unsigned long long nd, uint32_t s) {
    return (nd >> (kNdBits * (s - 1u))) & ((1ull << kNdBits) - 1ull);
}

// Code field of state(w_i, w_t), i < t, of a k = 5 pattern in the state-vector
// layout.
__device__ __forceinline__ constexpr uint32_t e5(int i, int t, uint32_t s) {
    return s << ((t == 1 ? 18 : t == 2 ? 14 : t == 3 ? 8 : 0) + 2 * i);
}

// Sums by k = 5 class: the low words in shared memory, the carries (and high
// words) straight to the global sums.
struct Bins5 {
    uint32_t *lo;  // num_classes(5) words
    unsigned long long *sums;
    const int16_t *lut;
    int *status;
    __device__ __forceinline__ void add_class(int c, unsigned long long d) const {
        const uint32_t l = (uint32_t)d;
        uint32_t hi = (uint32_t)(d >> 32);
        if (l) {
            const uint32_t old = atomicAdd(&lo[c], l);
            if (old > ~l) hi++;
        }
        if (hi) atomicAdd(&sums[c], (unsigned long long)hi << 32);
    }
    __device__ __forceinline__ void add(uint32_t code, unsigned long long d) const {
        const int c = (int)__ldg(lut + code);
        if (c < 0) set_status(status, ACC_ERR_INTERNAL);
        else add_class(c, d);
    }
    // whole block, a barrier on both sides
    __device__ __forceinline__ void clear() const {
        for (int i = threadIdx.x; i < num_classes(5); i += blockDim.x) lo[i] = 0u;
        __syncthreads();
    }
    __device__ __forceinline__ void flush() const {
        __syncthreads();
        for (int i = threadIdx.x; i < num_classes(5); i += blockDim.x)
            if (lo[i]) atomicAdd(&sums[i], (unsigned long long)lo[i]);
    }
};

// Common neighbours of the edge of entry p (row vertex x, neighbour y), typed
// word i field j by state i + 1 to x and j + 1 to y.
struct EdgeTri {
    unsigned long long w[3];
    bool flip;
    __device__ __forceinline__ bool any() const { return (w[0] | w[1] | w[2]) != 0ull; }
    __device__ __forceinline__ unsigned long long get(uint32_t i, uint32_t j) const {
        const uint32_t a = flip ? j : i, b = flip ? i : j;
        return nd_of(a == 0u ? w[0] : (a == 1u ? w[1] : w[2]), b + 1u);
    }
};
__device__ __forceinline__ EdgeTri edge_tri(const PartialArgs &a, long long p, bool upper) {
    const long long q = upper ? p : (long long)a.rev[p].x - 1;
    return EdgeTri{{a.tri[3 * q], a.tri[3 * q + 1], a.tri[3 * q + 2]}, !upper};
}

// k = 5: whether the list scan counts the set instead (or the build refused it).
__device__ __forceinline__ bool scan_flag(const PartialArgs &a) {
    return *(volatile unsigned long long *)(a.p5.ctr + kCtrScan) != 0ull ||
           (a.status && *(volatile int *)a.status == ACC_ERR_OVERFLOW);
}
// One answer for the whole block: thread 0 asks, and every thread reads it after the
// kernel's first barrier, before any other thread of the block may have left.  The
// flag may be raised while a kernel's blocks start, by the kernel itself or one beside
// it, and a warp that left while others of its block stayed would leave its share of
// the tables uncleared.  (The answer is on its way while the tables are cleared.)
__device__ __forceinline__ void ask_scan(const PartialArgs &a, int *instead) {
    if (threadIdx.x == 0) *instead = scan_flag(a);
}
__device__ __forceinline__ bool scan_instead(const PartialArgs &a) {
    __shared__ int instead;
    ask_scan(a, &instead);
    __syncthreads();
    return instead != 0;
}

// Nonzero types of an edge's common neighbours: bit 3 i + j for states i + 1 and
// j + 1 to the ends the edge is seen from.
__device__ __forceinline__ uint32_t types_of(const EdgeTri &t) {
    uint32_t m = 0;
#pragma unroll
    for (uint32_t i = 0; i < 3; i++)
#pragma unroll
        for (uint32_t j = 0; j < 3; j++)
            if (nd_of(t.w[i], j + 1u)) m |= 1u << (t.flip ? 3u * j + i : 3u * i + j);
    return m;
}
__device__ __forceinline__ uint32_t next_bit(uint32_t m) { return (uint32_t)__ffs((int)m) - 1u; }

// The matrix from partial counts to induced ones (k = 3, 4): the number of its
// entries, then (to << 24) | (from << 16) | (coefficient + 2^15).  lut,
// class_code: the class table in the canonical layout (host).
void partial_matrix(int k, const int16_t *lut, const uint32_t *class_code, std::vector<uint32_t> &out);

// Counts the built set (k = 3, 4; largest degree at most kNdMax) and clears
// its dense block; max_entries bounds 2 |E*|.  Returns the launches.
int launch_partial(int k, PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s, int grid_num = 1,
                   int grid_den = 1);

// k = 5, partial5.cu.  partial5_tables: divisors and automorphisms (host).
void partial5_tables(const uint32_t *code5, const uint32_t *code4, const uint32_t *code3, std::vector<unsigned char> &div5,
                     std::vector<unsigned char> &aut4, std::vector<unsigned char> &aut3);
// The sums of one built graph; then (after the scan's kernels, which run only
// when ctr[kCtrScan] is set) the counts from them.
int launch_partial5(PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s, int grid_num, int grid_den);
int launch_partial5_counts(const PartialArgs &a, int num_sms, cudaStream_t s);
// (partial.cu) typed degrees; 4-cycles and triangles by phase; the other partial
// counts of k = 4; the pair pass by phase.
int launch_partial5_prep(const PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s);
int launch_partial5_wedges(const PartialArgs &a, int phase, int num_sms, cudaStream_t s, int grid_num, int grid_den);
int launch_partial5_finish(PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s);
int launch_partial5_pairs(const PartialArgs &a, int phase, int num_sms, cudaStream_t s, int grid_num, int grid_den);

}  // namespace acc
