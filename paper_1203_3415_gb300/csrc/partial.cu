// Counting by partial patterns (k = 3, 4): the count mode of the larger sets
// (uses_partial) whose vertices are renumbered by descending degree.
//
// A partial pattern fixes the pair states of some pairs of a k-set (its
// edges, which connect the set) and leaves the other pairs open.  With P(c)
// the number of k-sets in which class c occurs as a partial pattern (each
// occurrence counted) and I(c) the induced count the library reports, a set
// of class c' contains c once for every subset of its G* edges whose pattern
// is c, so by inclusion and exclusion over the edges left out
//   I(c) = sum over c' and edge subsets S of c' with class(S) = c of
//          (-1)^(edges of c' - |S|) P(c').
// The partial counts need no walk over the k-sets, as the paper's set-size
// formulas do not (Table starb, Table ept): a path or a star is a product of
// typed degrees, a triangle with a pendant arc one of a typed triangle count
// and a degree, and what has to be visited is only
//   wedges v - u - w with v the smallest id (k = 4, for the 4-cycles: the
//   wedges of one v that end in the same w, by their two states),
//   triangles, and for the 4-cliques the common neighbours of a triangle.
// In degree order those are few: on 20000 vertices and 100000 arcs (Chung-Lu,
// degrees up to 500) 1.35e6 wedges and 1.5e4 triangles, where the scan of
// the extension lists (enum.cu) reads 8.6e7 entries.
//
// Every sum is exact modulo 2^64, and the reported counts are below 2^62.
#include <type_traits>

#include "common.cuh"
#include "partial.cuh"

namespace acc {

namespace {

constexpr int kPWarps = 8;           // warps per block
constexpr int kPThreads = kPWarps * kWarp;
// Wedge tables, 16 bytes a slot: one a warp for the roots with few wedges, one
// a block for the others (k = 5: smaller, beside the block's sums).
// A warp's table: of a set of graphs three times as many slots, at half the
// warps an SM.  A root on a warp takes less work than on a block, whose warps
// each have their fixed part, so where roots are plenty the warps keep those of
// up to 384 wedges: 4008 graphs, phases 1 + 2: 1.3 + 9.9 ms with 192 slots, 2.6 +
// 8.2 with 576.
constexpr int kSlots = 192, kSetSlots = 576;
__host__ __device__ constexpr int warp_fill(int slots) { return slots == kSetSlots ? 384 : 144; }  // most keys it takes
__host__ __device__ constexpr int block_slots(int K) { return K == 5 ? 1024 : 2048; }
__host__ __device__ constexpr int wide_slots(int K) { return block_slots(K) / 2; }  // 28-byte slots: key, three words of 21-bit counts
constexpr int kRowParts = 1024;      // k = 4: rows whose part of a range of ends is kept
constexpr int kFieldMax = 1023;      // largest count of a 16-byte slot's fields
constexpr int kRingP = 64;           // rows staged for the flat scan
constexpr int kRingArrays = 5;       // (k = 4: 4, the root is packed into the entry)
constexpr int kRoots = 16;           // roots that share a table pass
constexpr int kHits = 96;            // triangles held before they are counted, two words each
constexpr int kFThreads = 256;       // threads per block of the finish

// ---------------------------------------------------------------------------
// Preparation: typed degrees, and for k = 4 the reverse positions of the upper
// entries (v -> u with u above v: the part of N*(u) above v, as k_rev gives
// it for every entry), the wedges of each v, and cleared triangle counters.
// Thread per neighbour entry; bound by the dependent loads of its search (8 us at
// 1.9e5 entries).
// ---------------------------------------------------------------------------
template <int K>
__global__ void k_partial_prep(PartialArgs a) {
    grid_dep_wait();
    const long long nnz = a.info->nnz;
    const int lane = threadIdx.x & 31;
    if (K == 5 && blockIdx.x == 0 && threadIdx.x == 0 && a.info->to_scan) a.p5.ctr[kCtrScan] = 1ull;
    const bool hubs = K == 5 && a.info->maxdeg > kCycleRows;
    for (long long p0 = blockIdx.x * (long long)blockDim.x + threadIdx.x - lane; p0 < nnz;
         p0 += (long long)gridDim.x * blockDim.x) {
        const long long pos = p0 + lane;
        const bool ok = pos < nnz;
        const uint32_t r = ok ? a.src[pos] : 0xFFFFFFFFu, v = r & 0x7FFFFFFFu;
        const uint32_t e = ok ? a.nbr[pos] : 0u;
        // a row's entries sit on consecutive lanes: one add per row and warp
        // (an add per entry took 25 us at 1.9e5 entries: a hub row's adds meet
        // in one word)
        const unsigned same = __match_any_sync(kFull, (int)v);
        const bool leader = ok && lane == __ffs(same) - 1;
        const unsigned m1 = __ballot_sync(kFull, (e & 3u) == 1u), m2 = __ballot_sync(kFull, (e & 3u) == 2u),
                       m3 = __ballot_sync(kFull, (e & 3u) == 3u);
        if (leader)
            atomicAdd(&a.nd[v], (unsigned long long)__popc(same & m1) |
                                    ((unsigned long long)__popc(same & m2) << kNdBits) |
                                    ((unsigned long long)__popc(same & m3) << (2 * kNdBits)));
        // k = 5: a root with more rows than the 5-cycle tables count leaves the graph to
        // the scan.  Decided here, before the passes, so that they are not run for
        // nothing.
        if (K == 5 && hubs && leader && a.deg[v] - a.lo[v] > kCycleRows) a.p5.ctr[kCtrScan] = 1ull;
        if constexpr (K >= 4) {
            uint2 rv = make_uint2(0u, 0u);
            if (ok && (K == 5 || !(r >> 31))) {
                const int voff = a.gs.meta(a.gs.graph_of((int)v)).voff;
                const uint32_t u = (uint32_t)voff + (e >> 2);
                const long long base = a.nptr[u];
                // (k = 4: v is among the neighbours of u below u)
                const int i = lower_id(a.nbr + base, K == 5 ? a.deg[u] : a.lo[u], v - (uint32_t)voff);
                rv = make_uint2((uint32_t)(base + i + 1), (uint32_t)(a.deg[u] - i - 1));
                if (!(r >> 31))
#pragma unroll
                    for (int j = 0; j < 3; j++) a.tri[3 * pos + j] = 0ull;
            }
            if (ok) a.rev[pos] = rv;
            auto row_sum = [&](uint32_t x) -> uint32_t {  // of the row's lanes, seen from its first
                uint32_t incl = x;
#pragma unroll
                for (int d = 1; d < kWarp; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(kFull, incl, d);
                    if (lane >= d) incl += y;
                }
                const int last = lane + __popc(same >> lane) - 1;
                return __shfl_sync(kFull, incl, last) - incl + x;
            };
            const uint32_t sum = row_sum(r >> 31 ? 0u : rv.y);
            if (leader && sum) atomicAdd(&a.wedges[v], sum);
            if constexpr (K == 5) {
                if (leader && sum) atomicAdd(&a.p5.cycle_wedges[v], sum);
                const uint32_t all = row_sum(rv.y);
                if (leader && all) atomicAdd(&a.p5.pair_wedges[v], all);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Wedges and triangles
// ---------------------------------------------------------------------------

// A warp's working storage and the graph it counts.
template <int K, bool HASH>
struct Walker {
    static constexpr int kWideSlots = wide_slots(K);
    const PartialArgs *a;
    PView g;
    uint32_t *hist;   // this warp's histogram of partial counts (two words a class)
    Bins5 bins;       // k = 5: the block's sums
    uint4 *tab;       // k = 4, 5: (key, three words of three 10-bit counts)
    uint32_t slots;   // the table's slots
    const uint2 *parts = nullptr;  // the rows' parts of the range, from row parts0 on, or NULL
    long long parts0 = 0;
    uint32_t *ring;   // flat start, entry offset, row position, row entry[, row vertex]
    uint32_t *hq;     // k = 4: triangles held (positions of v -> u and u -> w)
    int held;
    int gcur;
    unsigned long long scanned;
    int lane;

    __device__ __forceinline__ int cls(uint32_t code) const { return (int)__ldg(a->lut + code); }
    __device__ __forceinline__ void add(uint32_t code, unsigned long long d) {
        if constexpr (K == 5) {
            bins.add(code, d);
            return;
        }
        const int c = cls(code);
        if (c < 0) set_status(a->status, ACC_ERR_INTERNAL);
        else hist_add(hist, c, d);
    }

    // the histogram into graph gcur's partial counts (whole warp)
    __device__ __forceinline__ void drain() {
        if constexpr (K == 5) return;  // (one graph; the block flushes its sums)
        constexpr int N = num_classes(K);
        if (K == 4 && held) triangles(held);
        held = 0;
        __syncwarp();
        if (gcur >= 0)
            for (int c = lane; c < N; c += kWarp) {
                const unsigned long long v =
                    (unsigned long long)hist[2 * c] | ((unsigned long long)hist[2 * c + 1] << 32);
                if (v) {
                    hist[2 * c] = hist[2 * c + 1] = 0u;
                    atomicAdd(&a->part[(size_t)gcur * N + c], v);
                }
            }
        __syncwarp();
    }

    __device__ __forceinline__ void switch_graph(int gi) {
        if (gi == gcur) return;
        drain();
        gcur = gi;
        g = pview(*a, a->gs.meta(gi));
    }

    // k = 4: the last n <= 32 triangles held (v < u < w), a lane each.  Each
    // edge's typed counter of common neighbours takes the third vertex (edge
    // b < c, common neighbour x: word state(b, x), field state(c, x)), and the
    // 4-cliques v < u < w < x are found among the neighbours of w above w: the
    // triangles' lists as one flat sequence, kAhead entries a lane in flight
    // (phase 2 of 20000 vertices, 1.5e4 triangles: 85 us; 190 us with a lane
    // walking its own triangle's list, which waits for one entry at a time).
    __device__ __forceinline__ void triangles(int n) {
        constexpr int kAhead = 4;
        __syncwarp();
        uint32_t v = 0, u = 0, code = 0, off = 0;
        int len = 0;
        if (lane < n) {
            const uint32_t pvu = hq[2 * (held - n + lane)], puw = hq[2 * (held - n + lane) + 1];
            const uint32_t e1 = __ldg(a->nbr + pvu), e2 = __ldg(a->nbr + puw), w = e2 >> 2;
            v = (__ldg(a->src + pvu) & 0x7FFFFFFFu) - (uint32_t)(g.deg - a->deg);
            u = e1 >> 2;
            const uint32_t svu = e1 & 3u, suw = e2 & 3u, svw = pstate<HASH>(g, v, w);
            const long long vb = g.nptr[v];
            const uint32_t pvw = (uint32_t)(vb + lower_id(a->nbr + vb, g.deg[v], w));
            atomicAdd(&a->tri[3ll * pvu + svw - 1u], 1ull << (kNdBits * (suw - 1u)));
            atomicAdd(&a->tri[3ll * pvw + svu - 1u], 1ull << (kNdBits * (swap_state(suw) - 1u)));
            atomicAdd(&a->tri[3ll * puw + swap_state(svu) - 1u], 1ull << (kNdBits * (swap_state(svw) - 1u)));
            code = (svu << 10) | ((svw | (suw << 2)) << 6);
            if (a->p5.tris) {  // counting k = 5: the triangle is listed
                const unsigned long long i = atomicAdd(&a->p5.ctr[kCtrTris], 1ull);
                if (i < a->p5.tri_cap) a->p5.tris[i] = make_uint4(pvu, puw, pvw, 0u);
                else a->p5.ctr[kCtrScan] = 1ull;
                a->p5.in_tri[v] = a->p5.in_tri[u] = a->p5.in_tri[w] = 1;
            }
            const int l = g.lo[w];
            off = (uint32_t)(g.nptr[w] + l);
            len = g.deg[w] - l;
        }
        int tot;
        const int pre = warp_excl(len, lane, &tot);
        off -= (uint32_t)pre;
        for (int t0 = 0; t0 < tot; t0 += kWarp * kAhead) {
            uint32_t x[kAhead], hv[kAhead], hu[kAhead], hc[kAhead], sv[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; i++) {
                const int t = t0 + i * kWarp + lane;
                int r = 0;  // the last triangle whose list starts at or before t
#pragma unroll
                for (int d = 16; d; d >>= 1)
                    if (__shfl_sync(kFull, pre, r + d) <= t) r += d;
                hv[i] = __shfl_sync(kFull, v, r);
                hu[i] = __shfl_sync(kFull, u, r);
                hc[i] = __shfl_sync(kFull, code, r);
                const uint32_t o = __shfl_sync(kFull, off, r);
                x[i] = t < tot ? __ldg(a->nbr + (o + (uint32_t)t)) : 0u;
            }
#pragma unroll
            for (int i = 0; i < kAhead; i++) sv[i] = x[i] ? pstate<HASH>(g, hv[i], x[i] >> 2) : 0u;
#pragma unroll
            for (int i = 0; i < kAhead; i++) {
                if (!sv[i]) continue;
                const uint32_t su = pstate<HASH>(g, hu[i], x[i] >> 2);
                if (su) add(hc[i] | sv[i] | (su << 2) | ((x[i] & 3u) << 4), 1ull);
            }
        }
        __syncwarp();
    }

    // One wedge end into the table: its key, the wedge's type (s1, s2).
    template <bool WIDE>
    __device__ __forceinline__ void put(uint32_t key, uint32_t s1, uint32_t s2) {
        constexpr int S = WIDE ? 1 : 4;  // words from one key to the next
        uint32_t *t = reinterpret_cast<uint32_t *>(tab);
        const uint32_t h = key * 0x9E3779B1u;
        uint32_t i = (uint32_t)(((unsigned long long)h * slots) >> 32);
        // (slots is 2^x or 3 2^x: 6 y + 1 steps through all of it)
        const uint32_t step = 6u * ((h >> 4) & 15u) + 1u;
        for (uint32_t tries = 0; tries < slots; tries++, i = i + step < slots ? i + step : i + step - slots) {
            const uint32_t old = atomicCAS(&t[S * i], 0u, key);
            if (old == 0u || old == key) {
                if constexpr (WIDE)
                    atomicAdd(reinterpret_cast<unsigned long long *>(t + kWideSlots) + 3 * i + (s1 - 1u),
                              1ull << (kNdBits * (s2 - 1u)));
                else
                    atomicAdd(&t[4 * i + s1], 1u << (10 * (s2 - 1u)));
                return;
            }
        }
        set_status(a->status, ACC_ERR_INTERNAL);  // (more keys than slots: the callers bound them)
    }

    // The slot that holds key, or -1.
    template <bool WIDE>
    __device__ __forceinline__ int find(uint32_t key) const {
        constexpr int S = WIDE ? 1 : 4;
        const uint32_t *t = reinterpret_cast<const uint32_t *>(tab);
        const uint32_t h = key * 0x9E3779B1u;
        uint32_t i = (uint32_t)(((unsigned long long)h * slots) >> 32);
        const uint32_t step = 6u * ((h >> 4) & 15u) + 1u;
        for (uint32_t tries = 0; tries < slots; tries++, i = i + step < slots ? i + step : i + step - slots) {
            const uint32_t k = t[S * i];
            if (k == key) return (int)i;
            if (!k) return -1;
        }
        return -1;
    }

    // Pairs of wedges with the same ends are 4-cycles v-b-w-d, typed by the
    // two wedges' states: field 3 (s1 - 1) + s2 - 1 of the three words w0, w1,
    // w2 (fields of B bits) counts the wedges of a type.
    template <int B, typename Word>
    __device__ __forceinline__ void cycles(Word w0, Word w1, Word w2) {
        constexpr Word mask = (Word(1) << B) - 1;
        uint32_t types = 0;
#pragma unroll
        for (int j = 0; j < 3; j++)
            types |= (((w0 >> (B * j)) & mask) ? 1u << j : 0u) | (((w1 >> (B * j)) & mask) ? 8u << j : 0u) |
                     (((w2 >> (B * j)) & mask) ? 64u << j : 0u);
        auto field = [&](uint32_t t) -> Word {
            const uint32_t i = t / 3u;
            const Word w = i == 0u ? w0 : (i == 1u ? w1 : w2);
            return (w >> (B * (t - 3u * i))) & mask;
        };
        for (uint32_t m = types; m; m &= m - 1u) {
            const uint32_t t = (uint32_t)__ffs((int)m) - 1u;
            const unsigned long long ct = field(t);
            const uint32_t c1 = ((t / 3u + 1u) << 10) | ((t % 3u + 1u) << 8);  // slots v, b, w
            for (uint32_t r = m; r; r &= r - 1u) {
                const uint32_t q = (uint32_t)__ffs((int)r) - 1u;
                const unsigned long long pairs = q == t ? ct * (ct - 1u) / 2 : ct * field(q);
                if (pairs) add(c1 | (q / 3u + 1u) | (swap_state(q % 3u + 1u) << 4), pairs);
            }
        }
    }

    // k = 5: the wedges of one pair {v, w} (words as above).  Three of them are
    // a K_{2,3}; two are a 4-cycle, and with a pendant at v or w a banner (its
    // other ends may coincide with the pendant; twice, as the cycle's two
    // middles may be swapped).
    template <int B, typename Word>
    __device__ __forceinline__ void pair_terms(Word w0, Word w1, Word w2, uint32_t v, uint32_t w) {
        constexpr Word mask = (Word(1) << B) - 1;
        uint32_t types = 0;
#pragma unroll
        for (int j = 0; j < 3; j++)
            types |= (((w0 >> (B * j)) & mask) ? 1u << j : 0u) | (((w1 >> (B * j)) & mask) ? 8u << j : 0u) |
                     (((w2 >> (B * j)) & mask) ? 64u << j : 0u);
        auto field = [&](uint32_t t) -> unsigned long long {
            const uint32_t i = t / 3u;
            const Word x = i == 0u ? w0 : (i == 1u ? w1 : w2);
            return (x >> (B * (t - 3u * i))) & mask;
        };
        auto middle = [](int m, uint32_t t) -> uint32_t {  // K_{2,3} with ends 0, 1
            return e5(0, m, t / 3u + 1u) | e5(1, m, swap_state(t % 3u + 1u));
        };
        const unsigned long long nv = g.nd[v], nw = g.nd[w];
        for (uint32_t m = types; m; m &= m - 1u) {
            const uint32_t t = (uint32_t)__ffs((int)m) - 1u;
            const unsigned long long ct = field(t);
            for (uint32_t r = m; r; r &= r - 1u) {
                const uint32_t q = (uint32_t)__ffs((int)r) - 1u;
                const unsigned long long cq = field(q), pairs = q == t ? ct * (ct - 1u) / 2 : ct * cq;
                if (!pairs) continue;
                const uint32_t cyc = e5(0, 1, t / 3u + 1u) | e5(1, 2, t % 3u + 1u) | e5(0, 3, q / 3u + 1u) |
                                     e5(2, 3, swap_state(q % 3u + 1u));
#pragma unroll
                for (uint32_t s = 1; s <= 3; s++) {
                    const unsigned long long xv = nd_of(nv, s), xw = nd_of(nw, s);
                    if (xv) add(cyc | e5(0, 4, s), 2u * pairs * xv);
                    if (xw) add(cyc | e5(2, 4, s), 2u * pairs * xw);
                }
                for (uint32_t z = r; z; z &= z - 1u) {
                    const uint32_t y = (uint32_t)__ffs((int)z) - 1u;
                    const unsigned long long cy = field(y);
                    unsigned long long n;
                    if (y == q) n = q == t ? (ct > 2 ? ct * (ct - 1u) / 2 * (ct - 2u) / 3 : 0ull) : ct * (cq * (cq - 1u) / 2);
                    else n = pairs * cy;
                    if (n) add(middle(2, t) | middle(3, q) | middle(4, y), n);
                }
            }
        }
    }

    // k = 5: houses.  A wedge v - b - w, another wedge v - d - w of the table,
    // and a common neighbour of v and b, or of b and w (which may coincide
    // with w or d, or v or d).  Rows as in scan, of the middles in a triangle.
    template <bool RANGED, bool WIDE>
    __device__ __forceinline__ void houses(long long p0, long long step, int nrows, uint32_t v0, uint32_t lo, uint32_t hi) {
        for (int jb = 0; jb < nrows; jb += kWarp) {
            const long long pl = p0 + (long long)(jb + lane) * step;
            int cl = 0;
            uint32_t fl = 0, el = 0;
            if (jb + lane < nrows) {
                el = __ldg(a->nbr + pl);
                if (a->p5.in_tri[el >> 2]) cl = row_part<RANGED>(pl, lo, hi, &fl);
            }
            for (unsigned rows = __ballot_sync(kFull, cl > 0); rows; rows &= rows - 1u) {
                const int r = __ffs(rows) - 1;
                const long long p = p0 + (long long)(jb + r) * step;
                const int cnt = __shfl_sync(kFull, cl, r);
                const uint32_t first = __shfl_sync(kFull, fl, r), e1 = __shfl_sync(kFull, el, r);
                const uint32_t src = __ldg(a->src + p), v = (src & 0x7FFFFFFFu), b = e1 >> 2, s1 = e1 & 3u;
                const EdgeTri tv = edge_tri(*a, p, !(src >> 31));
                const uint32_t mv = types_of(tv);
                for (int q = lane; q < cnt; q += kWarp) {
                    const uint32_t pos = first + (uint32_t)q, e2 = __ldg(a->nbr + pos), w = e2 >> 2, s2 = e2 & 3u;
                    const int i = find<WIDE>(((v - v0 + 1u) << 26) | w);
                    if (i < 0) continue;
                    const EdgeTri tw = edge_tri(*a, pos, b < w);
                    const uint32_t mw = types_of(tw);
                    if (!(mv | mw)) continue;
                    const uint32_t *t = reinterpret_cast<const uint32_t *>(tab);
                    auto count = [&](uint32_t y) -> unsigned long long {  // wedges of type y but this one
                        const uint32_t own = y == 3u * (s1 - 1u) + s2 - 1u ? 1u : 0u;
                        if constexpr (WIDE)
                            return nd_of(reinterpret_cast<const unsigned long long *>(t + kWideSlots)[3 * i + y / 3u], y % 3u + 1u) - own;
                        else
                            return ((t[4 * i + 1 + y / 3u] >> (10 * (y % 3u))) & 1023u) - own;
                    };
                    for (uint32_t y = 0; y < 9; y++) {
                        const unsigned long long c = count(y);
                        if (!c) continue;
                        const uint32_t cyc = e5(0, 1, s1) | e5(1, 2, s2) | e5(0, 3, y / 3u + 1u) |
                                             e5(2, 3, swap_state(y % 3u + 1u));
                        for (uint32_t m = mv; m; m &= m - 1u) {
                            const uint32_t z = next_bit(m);
                            add(cyc | e5(0, 4, z / 3u + 1u) | e5(1, 4, z % 3u + 1u), c * tv.get(z / 3u, z % 3u));
                        }
                        for (uint32_t m = mw; m; m &= m - 1u) {
                            const uint32_t z = next_bit(m);
                            add(cyc | e5(1, 4, z / 3u + 1u) | e5(2, 4, z % 3u + 1u), c * tw.get(z / 3u, z % 3u));
                        }
                    }
                }
            }
        }
    }

    // Count the terms of slots i0, i0 + step, ... (i0 by lane) and empty
    // them.  Most ends take one wedge: the others are gathered in the (idle)
    // ring and counted 32 at a time.
    template <bool WIDE>
    __device__ __forceinline__ void sweep(int i0, int step, uint32_t v0) {
        if constexpr (WIDE) {
            uint32_t *t = reinterpret_cast<uint32_t *>(tab);
            for (int i = i0; i < (int)slots; i += step) {
                if (!t[i]) continue;
                unsigned long long *w = reinterpret_cast<unsigned long long *>(t + kWideSlots) + 3 * i;
                if constexpr (K == 5) pair_terms<kNdBits>(w[0], w[1], w[2], v0 + (t[i] >> 26) - 1u, t[i] & 0x3FFFFFFu);
                else cycles<kNdBits>(w[0], w[1], w[2]);
                t[i] = 0u;
                w[0] = w[1] = w[2] = 0ull;
            }
        } else {
            constexpr int H = K == 5 ? 4 : 3;
            int kept = 0;  // slots gathered, H words each
            auto count = [&](const uint32_t *h) {
                if constexpr (K == 5) pair_terms<10>(h[0], h[1], h[2], v0 + (h[3] >> 26) - 1u, h[3] & 0x3FFFFFFu);
                else cycles<10>(h[0], h[1], h[2]);
            };
            for (int b = i0 - lane; b < (int)slots; b += step) {
                const int i = b + lane;  // (the tables hold a multiple of 32 slots)
                const uint4 q = tab[i];
                if (q.x) tab[i] = make_uint4(0u, 0u, 0u, 0u);
                const uint32_t s = q.y + q.z + q.w;
                const bool many = q.x && (s & 1023u) + ((s >> 10) & 1023u) + (s >> 20) != 1u;
                const unsigned mm = __ballot_sync(kFull, many);
                if (many) {
                    uint32_t *h = ring + H * (kept + __popc(mm & ((1u << lane) - 1u)));
                    h[0] = q.y;
                    h[1] = q.z;
                    h[2] = q.w;
                    if (K == 5) h[H - 1] = q.x;
                }
                kept += __popc(mm);
                __syncwarp();
                if (kept >= kWarp) {
                    kept -= kWarp;
                    count(ring + H * (kept + lane));
                    __syncwarp();
                }
            }
            if (lane < kept) count(ring + H * lane);
            __syncwarp();
        }
    }

    // The part of row entry p's list that the scan takes: k = 3 the
    // neighbours of u above u (triangles v < u < w); k = 4 those of u above
    // v, within [lo, hi) when RANGED.
    template <bool RANGED>
    __device__ __forceinline__ int row_part(long long p, uint32_t lo, uint32_t hi, uint32_t *first) const {
        if constexpr (K == 3) {
            const uint32_t r = __ldg(a->src + p);
            if (r >> 31) return 0;
            const uint32_t u = __ldg(a->nbr + p) >> 2;
            const int l = g.lo[u];
            *first = (uint32_t)(g.nptr[u] + l);
            return g.deg[u] - l;
        } else {
            if constexpr (RANGED && K == 4)
                if (parts) {
                    const uint2 x = parts[p - parts0];
                    *first = x.x;
                    return (int)x.y;
                }
            // (entries below the row's vertex lie between the rows of a shared pass)
            if (K == 4 && (__ldg(a->src + p) >> 31)) return 0;
            const uint2 r = __ldg(a->rev + p);
            *first = r.x;
            int cnt = (int)r.y;
            if constexpr (RANGED)
                if (cnt) cnt = id_range(a->nbr, cnt, lo, hi, first);
            return cnt;
        }
    }

    // Scan rows p0, p0 + step, ... (nrows of them) as one flat sequence of
    // 32-entry windows, a lane an entry, across row boundaries (the staging
    // and row lookup of enum.cu's count_leaves), two windows at a time.
    // k = 4: the rows' roots are v0, v0 + 1, ... (at most kRoots of them; one
    // when the end vertices are restricted to [lo, hi)).
    template <bool RANGED, bool WIDE>
    __device__ __forceinline__ void scan(long long p0, long long step, int nrows, uint32_t v0, uint32_t lo, uint32_t hi) {
        constexpr int RM = kRingP - 1;
        constexpr int W = 2;
        uint32_t *rS = ring, *rO = ring + kRingP, *rP = ring + 2 * kRingP, *rE = ring + 3 * kRingP,
                 *rV = ring + 4 * kRingP;
        uint32_t T = 0, F = 0;
        int tail = 0, cur = -1, jb = 0;
        const uint32_t voff = (uint32_t)(g.deg - a->deg);
        for (;;) {
            while (jb < nrows && T - F < 32u * W && tail - cur + kWarp <= kRingP) {
                const long long p = p0 + (long long)(jb + lane) * step;
                int cnt = 0;
                uint32_t first = 0;
                if (jb + lane < nrows) cnt = row_part<RANGED>(p, lo, hi, &first);
                const unsigned nz = __ballot_sync(kFull, cnt > 0);
                jb += kWarp;
                if (!nz) continue;
                int tot;
                const int pre = warp_excl(cnt, lane, &tot);
                if (cnt > 0) {
                    const int slot = (tail + __popc(nz & ((1u << lane) - 1u))) & RM;
                    const uint32_t sflat = T + (uint32_t)pre;
                    rS[slot] = sflat;
                    rO[slot] = first - sflat;
                    rP[slot] = (uint32_t)p;
                    const uint32_t v = (__ldg(a->src + p) & 0x7FFFFFFFu) - voff;
                    if (K == 3) {
                        rE[slot] = __ldg(a->nbr + p);
                        rV[slot] = v;
                    } else {
                        rE[slot] = __ldg(a->nbr + p) | ((v - v0) << 28);  // (ids have 26 bits)
                    }
                }
                tail += __popc(nz);
                T += (uint32_t)tot;
            }
            const uint32_t pend = T - F;
            if (!pend) break;
            __syncwarp();
            uint32_t v[W], e1[W], pvu[W], puw[W], e2[W], svw[W];
            bool ok[W];
#pragma unroll
            for (int w = 0; w < W; w++) {
                const uint32_t t0 = F + 32u * w;
                uint32_t bit = 0;
                const int r = cur + 1 + lane;
                if (r < tail) {
                    const uint32_t sd = rS[r & RM] - t0;
                    if (sd < 32u) bit = 1u << sd;
                }
                const uint32_t starts = __reduce_or_sync(kFull, bit);
                const int row = (cur + __popc(starts & (0xFFFFFFFFu >> (31 - lane)))) & RM;
                cur += __popc(starts);
                ok[w] = 32u * w + (uint32_t)lane < pend;
                e1[w] = rE[row];
                if (K == 3) {
                    v[w] = rV[row];
                } else {
                    v[w] = e1[w] >> 28;
                    e1[w] &= 0x0FFFFFFFu;
                }
                pvu[w] = rP[row];
                puw[w] = rO[row] + t0 + (uint32_t)lane;
                e2[w] = ok[w] ? __ldg(a->nbr + puw[w]) : 0u;
            }
#pragma unroll
            for (int w = 0; w < W; w++)
                svw[w] = K < 5 && ok[w] && (K == 3 || (e2[w] >> 2) > (e1[w] >> 2)) ? pstate<HASH>(g, K == 3 ? v[w] : v0 + v[w], e2[w] >> 2) : 0u;
            if constexpr (K >= 4) {
#pragma unroll
                for (int w = 0; w < W; w++)
                    if (ok[w])
                        put<WIDE>(((v[w] + 1u) << 26) | (e2[w] >> 2), e1[w] & 3u,
                                  e2[w] & 3u);
            }
            if constexpr (K < 5)
#pragma unroll
            for (int w = 0; w < W; w++) {
                const uint32_t e = (e1[w] & 3u) << 4 | svw[w] | (e2[w] & 3u) << 2;
                if constexpr (K == 3) {
                    if (svw[w]) add(e, 1ull);
                } else {
                    const unsigned m = __ballot_sync(kFull, svw[w] != 0u);
                    if (svw[w]) {
                        uint32_t *h = hq + 2 * (held + __popc(m & ((1u << lane) - 1u)));
                        h[0] = pvu[w];
                        h[1] = puw[w];
                    }
                    held += __popc(m);
                }
            }
            if constexpr (K == 4)
                while (held >= kWarp) {
                    triangles(kWarp);
                    held -= kWarp;
                }
            F += pend < 32u * W ? pend : 32u * W;
        }
        scanned += T;
    }
};

// k = 4.  Phase 1: up to 32 consecutive vertices a grab; roots with few wedges
// share passes over the warp's table (up to kFill wedges a pass), a root
// with more is queued in parts, ranges of end vertices that carry about
// equal neighbour entries (a wedge ends in w about in proportion to w's
// degree).  Phase 2: a block per part, whose warps fill one table of
// kBlockSlots slots; the rows are dealt to the warps one by one, since a
// root's first neighbours are hubs with the longest rows.
//
// Bound by the latency of list entry, state and table (L2, shared memory).
// A part re-reads the root's rows (two binary searches a row, side by side, and
// kept for the scan), so parts are as long as the table allows: on 20000 vertices
// and 1.35e6 wedges, parts of 160 wedges on one warp's table executed 83e6 warp
// instructions, this about 27e6.  Measured with blocks of 16 warps and 4096 slots
// / 4 and 1024 / 8 and 2048: 4008 graphs (1.4e8 wedges of such roots, 900 a root)
// 18.2 / 10.6 / 10.6 ms in phase 2, and the whole count of 10^6 vertices - /
// 3.64 / 3.09 ms.
//
// k = 5 runs the same passes over the wedges with any middle and the root as
// the smaller end (K_{2,3}, banners and houses), for one graph.
// (BESIDE: k = 4 counted for k = 5, beside the 5-cycles.)
template <int K, int PHASE, bool HASH, bool BESIDE, int SLOTS>
__global__ void __launch_bounds__(kPThreads, K == 5 ? 3 : (SLOTS == kSetSlots && PHASE == 1 ? 2 : 4)) k_wedges(PartialArgs a) {
    const typename std::conditional<BESIDE, JoinsPrevious, WaitsForPrevious>::type order;
    if (K == 5) grid_dep_launch();  // k_partial_finish, then k_vertex5 and its followers run beside
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int kSlots = SLOTS, kFill = warp_fill(SLOTS);
    __shared__ uint4 item;
    __shared__ uint32_t bounds[2];
    constexpr int kBlockSlots = block_slots(K), kBlockFill = kBlockSlots * 2 / 3, kWideFill = wide_slots(K) * 2 / 3,
                  kPart = kBlockFill * 7 / 8, kWidePart = kWideFill * 7 / 8;
    __shared__ unsigned long long sizes[kPWarps];
    constexpr int N = num_classes(4);
    unsigned long long *ctr = a.p5.ctr;
    // (counting k = 5, the scan's counters stay as the build left them)
    unsigned long long *unit = K == 5 ? ctr + kCtrPairUnit : (ctr ? ctr + kCtrUnit4 : &a.info->unit_ctr),
                       *qtail = K == 5 ? ctr + kCtrPairTail : (ctr ? ctr + kCtrTail4 : &a.info->queue_tail),
                       *qhead = K == 5 ? ctr + kCtrPairHead : (ctr ? ctr + kCtrHead4 : &a.info->queue_head);
    // (k = 5: the second half of the queue has the 5-cycles' parts)
    const unsigned long long queue_cap = ctr ? a.queue_cap / 2 : a.queue_cap;
    uint32_t *root_wedges = K == 5 ? a.p5.pair_wedges : a.wedges;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    if (a.status && *(volatile int *)a.status == ACC_ERR_OVERFLOW) return;
    __shared__ int instead;
    if (K == 5 || BESIDE) ask_scan(a, &instead);
    if (PHASE == 2 && *qtail == 0) return;
    uint4 *tabs = reinterpret_cast<uint4 *>(smem);
    Walker<K, HASH> wk;
    wk.a = &a;
    constexpr int kTab = PHASE == 1 ? kPWarps * kSlots : kBlockSlots;
    wk.tab = PHASE == 1 ? tabs + wib * kSlots : tabs;
    wk.slots = kSlots;
    uint32_t *words = reinterpret_cast<uint32_t *>(smem + kTab * 16);
    wk.ring = words + wib * kRingP * 4;
    wk.hq = words + kPWarps * kRingP * 4 + wib * 2 * kHits;
    // (one histogram a block when its warps are at one graph at a time: with
    // one a warp, 4864 warps add to the same few sums at the end)
    const bool one_hist = PHASE == 2 || K == 5 || a.gs.B == 1;
    wk.hist = words + kPWarps * (kRingP * 4 + (K == 4 ? 2 * kHits : 0)) + (one_hist ? 0 : wib * 2 * N);
    wk.bins = Bins5{wk.hist, a.p5.sums, a.p5.lut5, a.status};  // (k = 5: one histogram a block)
    uint2 *row_parts = reinterpret_cast<uint2 *>(wk.hist + (PHASE == 2 && K == 4 ? 2 * N : 0));
    wk.held = 0;
    wk.gcur = -1;
    wk.scanned = 0;
    wk.lane = lane;
    for (int i = threadIdx.x; i < kTab; i += kPThreads) tabs[i] = make_uint4(0u, 0u, 0u, 0u);
    if constexpr (K == 5) wk.bins.clear();
    else
        for (int i = lane; i < 2 * N; i += kWarp) wk.hist[i] = 0u;
    __syncthreads();
    if ((K == 5 || BESIDE) && instead) return;
    // first row of root v (k = 4: of the vertices above it)
    auto first_row = [&](uint32_t v) -> long long { return wk.g.nptr[v] + (K == 5 ? 0 : wk.g.lo[v]); };
    // parts of a root with W wedges and d rows
    auto parts_of = [](uint32_t W, int d) -> uint32_t {
        return d > kFieldMax ? (W <= (uint32_t)kWideFill ? 1u : (W + kWidePart - 1) / kWidePart)
                             : (W <= (uint32_t)kBlockFill ? 1u : (W + kPart - 1) / kPart);
    };
    if constexpr (PHASE == 1) {
        // vertices a grab: up to 32, and at least four grabs a warp (neighbouring
        // roots are similar work, and a warp takes them pass after pass)
        const long long warps = 4ll * gridDim.x * kPWarps;
        const int grab = (int)min(max((a.gs.NV + warps - 1) / warps, 1ll), (long long)kWarp);
        for (;;) {
            unsigned long long u0 = 0;
            if (lane == 0) u0 = atomicAdd(unit, (unsigned long long)grab);
            u0 = __shfl_sync(kFull, u0, 0);
            if ((long long)u0 >= a.gs.NV) break;
            const long long vg = (long long)u0 + lane;
            uint32_t W = 0;
            int gi = 0;
            if (lane < grab && vg < a.gs.NV) {
                W = root_wedges[vg];
                if (W) gi = a.gs.graph_of((int)vg);
            }
            const bool big = W > (uint32_t)kFill;
            const unsigned heavy = __ballot_sync(kFull, big);
            if (heavy) {
                // (a queued root's count is cleared: what the queue could not
                // take is found by its count at the end of phase 2)
                const uint32_t parts = big ? parts_of(W, a.deg[vg] - (K == 5 ? 0 : a.lo[vg])) : 0u;
                int tot;
                const int pre = warp_excl((int)parts, lane, &tot);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(qtail, (unsigned long long)tot);
                base = __shfl_sync(kFull, base, 0) + (unsigned long long)pre;
                if (base + parts <= queue_cap) {
                    for (uint32_t c = 0; c < parts; c++)
                        a.queue[base + c] = make_uint4((uint32_t)vg, parts == 1u ? W : c, parts, (uint32_t)gi);
                    if (parts) root_wedges[vg] = 0u;
                } else {
                    for (uint32_t c = 0; c < parts; c++)
                        if (base + c < queue_cap) a.queue[base + c] = make_uint4(0u, 0u, 0u, 0u);
                }
            }
            unsigned todo = __ballot_sync(kFull, W > 0u) & ~heavy;
            while (todo) {
                // the roots from the first one on, of one graph, up to the next
                // queued root and kFill wedges
                const int s = __ffs(todo) - 1;
                const int gs = __shfl_sync(kFull, gi, s);
                const unsigned after = heavy & ~((1u << s) - 1u);
                const int lim = after ? __ffs(after) - 1 : kWarp;
                const bool in = ((todo >> lane) & 1u) && gi == gs && lane < lim && lane < s + kRoots;
                int tot;
                const int pre = warp_excl(in ? (int)W : 0, lane, &tot);
                const bool ok = in && pre + (int)W <= kFill;
                const unsigned take = __ballot_sync(kFull, ok);
                const int e = __reduce_max_sync(kFull, ok ? lane : 0);
                wk.switch_graph(gs);
                const uint32_t voff = (uint32_t)a.gs.meta(gs).voff, v0 = (uint32_t)u0 + s - voff,
                               v1 = (uint32_t)u0 + e - voff;
                const long long p0 = first_row(v0), p1 = wk.g.nptr[v1] + wk.g.deg[v1];
                wk.template scan<false, false>(p0, 1, (int)(p1 - p0), v0, 0u, 0u);
                __syncwarp();
                if constexpr (K == 5)
                    if (ctr[kCtrTris]) {
                        wk.template houses<false, false>(p0, 1, (int)(p1 - p0), v0, 0u, 0u);
                        __syncwarp();
                    }
                wk.template sweep<false>(lane, kWarp, v0);
                __syncwarp();
                todo &= ~take;
            }
        }
    } else {
        // part `part` of `parts` of global root vg of graph gi, W wedges when
        // it is the only one (whole block)
        auto run_part = [&](uint32_t vg, uint32_t W, uint32_t part, uint32_t parts, int gi) {
            if (gi != wk.gcur) {
                // every warp's triangles are counted before the histogram moves on
                if constexpr (K == 4)
                    if (wk.held) wk.triangles(wk.held);
                wk.held = 0;
                __syncthreads();
                if (wib == 0) wk.drain();
                wk.gcur = gi;
                wk.g = pview(a, a.gs.meta(gi));
                __syncthreads();
            }
            const uint32_t v = vg - (uint32_t)(wk.g.deg - a.deg), n = (uint32_t)wk.g.n;
            const long long pb = first_row(v);
            const int rows = (int)(wk.g.nptr[v] + wk.g.deg[v] - pb);
            const bool wide = rows > kFieldMax;
            const uint32_t fill = wide ? kWideFill : kBlockFill;
            const long long p0 = pb + wib;
            const int nr = rows > wib ? (rows - wib + kPWarps - 1) / kPWarps : 0;
            // one pass over the root's rows, of at most `keys` distinct ends
            auto pass = [&](auto ranged, uint32_t keys, uint32_t lo, uint32_t hi) {
                constexpr bool R = decltype(ranged)::value;
                // the least of 192, 256, 384, ... that is at most two thirds full
                uint32_t sl = 192;
                while (2u * sl < 3u * keys) sl = sl % 3u ? sl + sl / 2u : sl / 3u * 4u;
                wk.slots = sl;
                if (wide) wk.template scan<R, true>(p0, kPWarps, nr, v, lo, hi);
                else wk.template scan<R, false>(p0, kPWarps, nr, v, lo, hi);
                __syncthreads();
                if constexpr (K == 5)
                    if (ctr[kCtrTris]) {
                        if (wide) wk.template houses<R, true>(p0, kPWarps, nr, v, lo, hi);
                        else wk.template houses<R, false>(p0, kPWarps, nr, v, lo, hi);
                        __syncthreads();
                    }
                if (wide) wk.template sweep<true>(threadIdx.x, kPThreads, v);
                else wk.template sweep<false>(threadIdx.x, kPThreads, v);
                __syncthreads();
            };
            // (a range's wedges may all end in one vertex: its counts fit the
            // fields, each at most the root's rows)
            if (parts == 1u) {
                pass(std::false_type{}, W < n ? W : n, 0u, 0u);
                return;
            }
            // ends [bound(part), bound(part + 1)): bound(c) is the first vertex
            // after v whose entries start at that share of the entries after v's
            if (threadIdx.x < 2) {
                const uint32_t c = part + threadIdx.x;
                const long long q0 = wk.g.nptr[v + 1], q1 = wk.g.nptr[n];
                const long long want = q0 + (q1 - q0) * (long long)c / (long long)parts;
                uint32_t x = v + 1u, y = n;
                if (c == 0) y = x;
                if (c == parts) x = y;
                while (x < y) {
                    const uint32_t mid = (x + y) >> 1;
                    if (wk.g.nptr[mid] < want) x = mid + 1u;
                    else y = mid;
                }
                bounds[threadIdx.x] = x;
            }
            __syncthreads();
            uint32_t lo = bounds[0], end = bounds[1];
            const uint32_t hi = end;
            while (lo < hi) {
                // wedges that end in [lo, end); when they and their ends are
                // more than the table takes, the range is halved
                const uint32_t width = end - lo;
                unsigned long long S = 0;
                wk.parts = nullptr;
                for (int r = threadIdx.x; r < rows; r += kPThreads) {
                    uint32_t first = 0;
                    const int cnt = wk.template row_part<true>(pb + r, lo, end, &first);
                    if (K == 4 && rows <= kRowParts) row_parts[r] = make_uint2(first, (uint32_t)cnt);
                    S += (unsigned long long)cnt;
                }
                if (K == 4 && rows <= kRowParts) {
                    wk.parts = row_parts;
                    wk.parts0 = pb;
                }
#pragma unroll
                for (int d = 16; d; d >>= 1) S += __shfl_xor_sync(kFull, S, d);
                if (lane == 0) sizes[wib] = S;
                __syncthreads();
                S = 0;
                for (int w = 0; w < kPWarps; w++) S += sizes[w];
                __syncthreads();
                const unsigned long long keys = S < width ? S : width;
                if (keys > fill) {
                    end = lo + width / 2;
                    continue;
                }
                if (S) pass(std::true_type{}, (uint32_t)keys, lo, end);
                lo = end;
                end = hi - lo > 2u * width ? lo + 2u * width : hi;
            }
        };
        const unsigned long long pushed = *qtail, tail = min(pushed, queue_cap);
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) {
                const unsigned long long idx = atomicAdd(qhead, 1ull);
                item = idx < tail ? a.queue[idx] : make_uint4(0xFFFFFFFFu, 0u, 0u, 0u);
            }
            __syncthreads();
            const uint4 it = item;
            if (it.x == 0xFFFFFFFFu) break;
            if (it.z) run_part(it.x, it.y, it.y, it.z, (int)it.w);
        }
        if (pushed > queue_cap) {
            for (long long vg = blockIdx.x; vg < a.gs.NV; vg += gridDim.x)
                for (uint32_t c = 0; c < 2u && root_wedges[vg] > (uint32_t)kFill; c++)
                    run_part((uint32_t)vg, 0u, c, 2u, a.gs.graph_of((int)vg));
        }
    }
    if (one_hist) {
        if constexpr (K == 4)
            if (wk.held) wk.triangles(wk.held);
        wk.held = 0;
        __syncthreads();
    }
    if constexpr (K == 5) {
        wk.bins.flush();
    } else {
        if (one_hist) wk.gcur = PHASE == 1 ? 0 : wk.gcur;
        if (!one_hist || wib == 0) wk.drain();
    }
    if (lane == 0 && wk.scanned) atomicAdd(&a.info->scanned, wk.scanned);
}

// k = 3: the triangles, 32 rows (neighbour entries) a grab.  The rows of one
// graph are dealt out with a stride, so that the hubs' rows, which come first
// and are the longest, end up in different grabs; a set of several graphs
// takes consecutive entries (few graph switches).  50000 vertices, 3.1e6 entries:
// 41 us (202 with consecutive rows; the two scan phases took 101), bound by the
// latency of entry and state.
template <bool HASH>
__global__ void __launch_bounds__(kPThreads, 4) k_partial3(PartialArgs a) {
    grid_dep_wait();
    constexpr int N = num_classes(3);
    __shared__ uint32_t rings[kPWarps][kRingP * kRingArrays];
    __shared__ uint32_t hists[kPWarps][2 * N];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    if (a.status && *(volatile int *)a.status == ACC_ERR_OVERFLOW) return;
    Walker<3, HASH> wk;
    wk.a = &a;
    wk.tab = nullptr;
    wk.slots = 0;
    wk.hq = nullptr;
    wk.held = 0;
    wk.ring = rings[wib];
    wk.hist = hists[wib];
    wk.gcur = -1;
    wk.scanned = 0;
    wk.lane = lane;
    if (lane < 2 * N) wk.hist[lane] = 0u;
    __syncwarp();
    const long long nnz = a.info->nnz, units = (nnz + kWarp - 1) / kWarp;
    for (;;) {
        unsigned long long q = 0;
        if (lane == 0) q = atomicAdd(&a.info->unit_ctr, 1ull);
        q = __shfl_sync(kFull, q, 0);
        if ((long long)q >= units) break;
        if (a.gs.B == 1) {
            wk.switch_graph(0);
            wk.template scan<false, false>((long long)q, units, (int)((nnz - (long long)q + units - 1) / units), 0u, 0u, 0u);
            continue;
        }
        const long long end = min(((long long)q + 1) * kWarp, nnz);
        for (long long p = (long long)q * kWarp; p < end;) {
            wk.switch_graph(a.gs.graph_of((int)(a.src[p] & 0x7FFFFFFFu)));
            const long long e = min(end, wk.g.nptr[wk.g.n]);
            wk.template scan<false, false>(p, 1, (int)(e - p), 0u, 0u, 0u);
            p = e;
        }
    }
    wk.drain();
    if (lane == 0 && wk.scanned) atomicAdd(&a.info->scanned, wk.scanned);
}

// ---------------------------------------------------------------------------
// Finish: the partial counts that are products of degrees and triangle
// counters, then the induced counts.
// ---------------------------------------------------------------------------

// Adds a per-thread sum to one class of the block's histogram (whole warp).
__device__ __forceinline__ void warp_add(uint32_t *hist, const int16_t *lut, int lane, uint32_t code,
                                         unsigned long long x) {
#pragma unroll
    for (int d = 16; d; d >>= 1) x += __shfl_xor_sync(kFull, x, d);
    if (lane == 0 && x) hist_add(hist, lut[code], x);
}

// One undirected edge b - c of G*, seen from the end where its state is 1 or 3:
// its state s, the neighbours of b other than c and of c other than b by state.
struct EdgeEnds {
    uint32_t s;
    bool flip;
    uint32_t b[3], c[3];  // (32 bits: their products are one wide multiply each)
};

__device__ __forceinline__ EdgeEnds edge_ends(uint32_t s, unsigned long long nb, unsigned long long nc) {
    EdgeEnds x;
    x.flip = s == 2u;
    x.s = x.flip ? 1u : s;
    const uint32_t r = swap_state(x.s);
    const unsigned long long n0 = x.flip ? nc : nb, n1 = x.flip ? nb : nc;
#pragma unroll
    for (uint32_t i = 0; i < 3; i++) {
        x.b[i] = (uint32_t)nd_of(n0, i + 1u) - (x.s == i + 1u ? 1u : 0u);
        x.c[i] = (uint32_t)nd_of(n1, i + 1u) - (r == i + 1u ? 1u : 0u);
    }
    return x;
}

// The terms of an edge with common neighbours (t: their counts by state to the
// ends the edge is seen from) that involve their kth nonzero type: paths that
// close (taken out), diamonds on the edge with a type not before it, and
// triangles on the edge with a pendant at one end (each of those seen from two
// edges: these counts are twice the real ones).
__device__ __forceinline__ void edge_triangles(uint32_t *hist, const int16_t *lut, const EdgeEnds &x, const EdgeTri &t,
                                               int kth) {
    const uint32_t f1 = x.s << 10;
    uint32_t m = types_of(t);
    for (int i = 0; i < kth; i++) m &= m - 1u;
    const uint32_t z = next_bit(m), i = z / 3u, j = z % 3u;
    const unsigned long long n = t.get(i, j);
    hist_add(hist, lut[f1 | ((i + 1u) << 6) | ((j + 1u) << 2)], 0ull - n);
    const uint32_t code = f1 | (((i + 1u) | ((j + 1u) << 2)) << 6);
    for (uint32_t r = m; r; r &= r - 1u) {
        const uint32_t q = next_bit(r);
        const unsigned long long pairs = q == z ? n * (n - 1u) / 2 : n * t.get(q / 3u, q % 3u);
        if (pairs) hist_add(hist, lut[code | (q / 3u + 1u) | ((q % 3u + 1u) << 2)], pairs);
    }
#pragma unroll
    for (uint32_t e = 0; e < 3; e++) {
        const unsigned long long xb = n * (x.b[e] - (e == i ? 1u : 0u)), xc = n * (x.c[e] - (e == j ? 1u : 0u));
        if (xb) hist_add(hist, lut[code | (e + 1u)], xb);
        if (xc) hist_add(hist, lut[code | ((e + 1u) << 2)], xc);
    }
}

// Induced counts of one graph from its partial counts (whole block), by the
// entries of partial_matrix.
template <int K>
__device__ void induced(const PartialArgs &a, int g, uint32_t *res, unsigned long long *P) {
    constexpr int N = num_classes(K);
    for (int i = threadIdx.x; i < 2 * N; i += blockDim.x) res[i] = 0u;
    // (read past the L1: other blocks wrote these sums)
    for (int i = threadIdx.x; i < N; i += blockDim.x) P[i] = atomicAdd(&a.part[(size_t)g * N + i], 0ull);
    __syncthreads();
    const int entries = (int)__ldg(a.inv);
#pragma unroll 4
    for (int i = threadIdx.x; i < entries; i += blockDim.x) {
        const uint32_t e = __ldg(a.inv + 1 + i);
        const unsigned long long x = P[(e >> 16) & 255u];
        if (x) hist_add(res, (int)(e >> 24), x * (unsigned long long)((long long)(e & 0xFFFFu) - 32768ll));
    }
    __syncthreads();
    for (int c = threadIdx.x; c < N; c += blockDim.x) {
        const unsigned long long x = (unsigned long long)res[2 * c] | ((unsigned long long)res[2 * c + 1] << 32);
        a.counts[(size_t)g * N + c] = K == 4 ? x >> 1 : x;  // (k = 4: twice the counts, see partial_matrix)
    }
    __syncthreads();
}

// 20000 vertices: 43 us cold (2.8 ms with slices of vertices, 88 with an edge a lane
// in its triangle terms), bound by the chain from an edge's degrees and triangle
// counts to the last block's matrix; a set of 4008 graphs 3.0 ms.
// Block per (graph, slice of its vertices and edges); the block that ends a
// graph's last slice turns the partial counts into induced ones.  On the
// dense block it also zeroes the marked chunks (k_clear_chunks).
template <int K, bool INDUCED>
__global__ void __launch_bounds__(kFThreads, 3) k_partial_finish(PartialArgs a) {
    const typename std::conditional<INDUCED, WaitsForPrevious, JoinsPrevious>::type order;  // (beside k_wedges<5, 1>)
    constexpr int N = num_classes(K);
    __shared__ uint32_t hist[2 * N];
    __shared__ unsigned long long sums[N];
    __shared__ uint32_t lists[kFThreads / kWarp][2 * kWarp];
    __shared__ __align__(16) int16_t lut_s[1 << code_bits(K)];
    __shared__ int last;
    const int lane = threadIdx.x & 31;
    if (!INDUCED && scan_instead(a)) return;
    if ((long long)blockIdx.x < (long long)a.gs.B * a.slices)
        for (int i = threadIdx.x; i < (1 << code_bits(K)) / 8; i += blockDim.x)
            reinterpret_cast<uint4 *>(lut_s)[i] = __ldg(reinterpret_cast<const uint4 *>(a.lut) + i);
    const bool refused = a.status && *(volatile int *)a.status == ACC_ERR_OVERFLOW;
    for (long long item = blockIdx.x; !refused && item < (long long)a.gs.B * a.slices; item += gridDim.x) {
        const int g = (int)(item / a.slices), sl = (int)(item % a.slices);
        const GMeta mt = a.gs.meta(g);
        for (int i = threadIdx.x; i < 2 * N; i += blockDim.x) hist[i] = 0u;
        __syncthreads();
        // stars (k = 3: the open triples) from the typed degrees
        const int v0 = (int)((long long)mt.n * sl / a.slices), v1 = (int)((long long)mt.n * (sl + 1) / a.slices);
        unsigned long long st[10] = {};
        for (int v = v0 + (int)threadIdx.x; v < v1; v += blockDim.x) {
            const unsigned long long nd = a.nd[mt.voff + v];
            const unsigned long long n1 = nd_of(nd, 1u), n2 = nd_of(nd, 2u), n3 = nd_of(nd, 3u);
            const unsigned long long p1 = n1 * (n1 - 1) / 2, p2 = n2 * (n2 - 1) / 2, p3 = n3 * (n3 - 1) / 2;
            if (K == 3) {
                st[0] += p1;
                st[1] += p2;
                st[2] += p3;
                st[3] += n1 * n2;
                st[4] += n1 * n3;
                st[5] += n2 * n3;
            } else {
                // (n (n - 1) / 2 is 0 for n = 0 modulo 2^64 too: n - 1 wraps and 0 times it is 0)
                st[0] += n1 > 2 ? n1 * (n1 - 1) / 2 * (n1 - 2) / 3 : 0ull;
                st[1] += n2 > 2 ? n2 * (n2 - 1) / 2 * (n2 - 2) / 3 : 0ull;
                st[2] += n3 > 2 ? n3 * (n3 - 1) / 2 * (n3 - 2) / 3 : 0ull;
                st[3] += p1 * n2;
                st[4] += p1 * n3;
                st[5] += p2 * n1;
                st[6] += p2 * n3;
                st[7] += p3 * n1;
                st[8] += p3 * n2;
                st[9] += n1 * n2 * n3;
            }
        }
        if (K == 3) {
            const uint32_t f[6] = {0x11, 0x22, 0x33, 0x12, 0x13, 0x23};  // (slot 1, slot 2) states
#pragma unroll
            for (int i = 0; i < 6; i++) warp_add(hist, lut_s, lane, ((f[i] >> 4) << 4) | (f[i] & 15u), st[i]);
        } else {
            const uint32_t f[10] = {0x111, 0x222, 0x333, 0x112, 0x113, 0x221, 0x223, 0x331, 0x332, 0x123};
#pragma unroll
            for (int i = 0; i < 10; i++)
                warp_add(hist, lut_s, lane, ((f[i] >> 8) << 10) | (((f[i] >> 4) & 15u) << 6) | (f[i] & 15u), st[i]);
            // paths, diamonds and triangles with a pendant from the edges
            unsigned long long p4[18] = {};
            // (slices of entries, not of vertices: a hub's row is as long as many others)
            const long long b0 = a.nptr[mt.voff], nb = a.nptr[mt.voff + mt.n] - b0;
            const long long e0 = b0 + nb * sl / a.slices, e1 = b0 + nb * (sl + 1) / a.slices;
            // edges with common neighbours are few in a sparse graph: a warp
            // gathers them, and takes 32 at a time by their (edge, type) pairs
            // (a lane an edge waited for up to a hundred adds one by one)
            uint32_t *list = lists[threadIdx.x >> 5];
            int kept = 0;
            auto edge_at = [&](uint32_t at, EdgeEnds *x) -> EdgeTri {
                const long long pos = e0 + at;
                const uint32_t e = a.nbr[pos];
                *x = edge_ends(e & 3u, a.nd[a.src[pos]], a.nd[mt.voff + (e >> 2)]);
                EdgeTri t = edge_tri(a, pos, true);
                t.flip = x->flip;
                return t;
            };
            auto closed = [&](int n) {  // the last n <= 32 gathered
                __syncwarp();
                EdgeEnds x;
                const int own = lane < n ? __popc(types_of(edge_at(list[kept - n + lane], &x))) : 0;
                int tot;
                const int pre = warp_excl(own, lane, &tot);
                for (int q0 = 0; q0 < tot; q0 += kWarp) {
                    const int q = q0 + lane;
                    int r = 0;
#pragma unroll
                    for (int d = 16; d; d >>= 1)
                        if (__shfl_sync(kFull, pre, r + d) <= q) r += d;
                    const int k = q - __shfl_sync(kFull, pre, r);
                    if (q < tot) {
                        const EdgeTri t = edge_at(list[kept - n + r], &x);
                        edge_triangles(hist, lut_s, x, t, k);
                    }
                }
                __syncwarp();
            };
            for (long long w0 = e0 + threadIdx.x - lane; w0 < e1; w0 += blockDim.x) {
                const long long pos = w0 + lane;
                const uint32_t r = pos < e1 ? a.src[pos] : 0x80000000u;
                bool tri = false;
                if (!(r >> 31)) {  // each edge once, from its smaller end
                    const uint32_t e = a.nbr[pos];
                    const EdgeEnds x = edge_ends(e & 3u, a.nd[r], a.nd[mt.voff + (e >> 2)]);
                    tri = (a.tri[3 * pos] | a.tri[3 * pos + 1] | a.tri[3 * pos + 2]) != 0ull;
#pragma unroll
                    for (int i = 0; i < 3; i++)
#pragma unroll
                        for (int j = 0; j < 3; j++) {
                            const unsigned long long y = (unsigned long long)x.b[i] * x.c[j];
                            p4[3 * i + j] += x.s == 3u ? 0ull : y;
                            p4[9 + 3 * i + j] += x.s == 3u ? y : 0ull;
                        }
                }
                const unsigned mm = __ballot_sync(kFull, tri);
                if (tri) list[kept + __popc(mm & ((1u << lane) - 1u))] = (uint32_t)(pos - e0);
                kept += __popc(mm);
                if (kept >= kWarp) {
                    closed(kWarp);
                    kept -= kWarp;
                }
            }
            closed(kept);
#pragma unroll
            for (uint32_t i = 0; i < 18; i++)
                warp_add(hist, lut_s, lane, ((i < 9 ? 1u : 3u) << 10) | (((i % 9) / 3 + 1u) << 6) | ((i % 3 + 1u) << 2),
                         p4[i]);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < N; c += blockDim.x) {
            const unsigned long long x = (unsigned long long)hist[2 * c] | ((unsigned long long)hist[2 * c + 1] << 32);
            if (x) atomicAdd(&a.part[(size_t)g * N + c], x);
        }
        if (!INDUCED) {  // (k = 5 reads the partial counts)
            __syncthreads();
            continue;
        }
        fence_device();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&a.done[g], 1) == a.slices - 1;
        __syncthreads();
        if (last) {
            fence_device();
            induced<K>(a, g, hist, sums);
        }
        __syncthreads();
    }
    if (INDUCED && a.occ)
        clear_chunks(a.gs, a.state_w, a.occ, a.occ_w, blockIdx.x * (long long)blockDim.x + threadIdx.x,
                     (long long)gridDim.x * blockDim.x);
}

bool launched() {
    if (cudaPeekAtLastError() == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

// Dynamic shared memory of k_wedges.
constexpr size_t wedge_smem(int K, int phase, int slots) {
    return (phase == 1 ? kPWarps * slots : block_slots(K)) * 16 + kPWarps * (kRingP * 16 + (K == 4 ? 8 * kHits : 0)) +
           (K == 5 ? 4 * num_classes(5) : (phase == 1 ? kPWarps : 1) * 8 * num_classes(4)) +
           (phase == 2 && K == 4 ? 8 * kRowParts : 0);
}

// The persistent grid times grid_num / grid_den, at least a block per SM.
int scaled_grid(int per_sm, int num_sms, int grid_num, int grid_den) {
    const long long g = (long long)num_sms * per_sm * grid_num / grid_den;
    return (int)(g < num_sms ? num_sms : g);
}

template <int K, int PHASE, bool HASH, bool BESIDE, int SLOTS = kSlots>
int wedge_phase(const PartialArgs &a, int num_sms, cudaStream_t s, int grid_num, int grid_den) {
    static std::atomic<unsigned long long> limit{0};
    if (!raise_shared_limit(k_wedges<K, PHASE, HASH, BESIDE, SLOTS>, wedge_smem(K, PHASE, SLOTS), limit)) return ACC_ERR_CUDA;
    // (no kernel waits on another block, so the grid need not be resident as a whole)
    const int grid = scaled_grid(K == 5 ? 3 : (SLOTS == kSetSlots && PHASE == 1 ? 2 : 4), num_sms, grid_num, grid_den);
    launch_pdl(k_wedges<K, PHASE, HASH, BESIDE, SLOTS>, grid, kPThreads, wedge_smem(K, PHASE, SLOTS), s, a);
    return launched() ? 1 : ACC_ERR_CUDA;
}

template <int K, bool BESIDE>
int wedges(const PartialArgs &a, int phase, int num_sms, cudaStream_t s, int grid_num, int grid_den) {
    if constexpr (K == 4 && !BESIDE) {
        if (a.gs.B > 1 && a.nh)
            return phase == 1 ? wedge_phase<K, 1, true, BESIDE, kSetSlots>(a, num_sms, s, grid_num, grid_den)
                              : wedge_phase<K, 2, true, BESIDE, kSetSlots>(a, num_sms, s, grid_num, grid_den);
        if (a.gs.B > 1)
            return phase == 1 ? wedge_phase<K, 1, false, BESIDE, kSetSlots>(a, num_sms, s, grid_num, grid_den)
                              : wedge_phase<K, 2, false, BESIDE, kSetSlots>(a, num_sms, s, grid_num, grid_den);
    }
    if (a.nh)
        return phase == 1 ? wedge_phase<K, 1, true, BESIDE>(a, num_sms, s, grid_num, grid_den)
                          : wedge_phase<K, 2, true, BESIDE>(a, num_sms, s, grid_num, grid_den);
    return phase == 1 ? wedge_phase<K, 1, false, BESIDE>(a, num_sms, s, grid_num, grid_den)
                      : wedge_phase<K, 2, false, BESIDE>(a, num_sms, s, grid_num, grid_den);
}

int grid_prep(long long max_entries, int num_sms) {
    long long grid = (max_entries + 255) / 256;
    if (grid > (long long)num_sms * 8) grid = (long long)num_sms * 8;
    return (int)(grid < 1 ? 1 : grid);
}

// Blocks of the finish, its slices of a graph: about four blocks per SM over
// the set, of at least 512 entries each.
int finish_grid(PartialArgs &a, long long max_entries, int num_sms) {
    long long sl = (4ll * num_sms + a.gs.B - 1) / a.gs.B;
    const long long per = max_entries / a.gs.B / 512 + 1;
    if (sl > per) sl = per;
    a.slices = (int)(sl < 1 ? 1 : sl);
    long long fin = (long long)a.gs.B * a.slices;
    const long long rows = (a.gs.NV * kWarp + kFThreads - 1) / kFThreads;  // (to clear them)
    if (a.occ && fin < rows) fin = rows;
    if (fin > (long long)num_sms * 8) fin = (long long)num_sms * 8;
    return (int)fin;
}

}  // namespace

// k = 4: a partial count of a triangle with a pendant is kept doubled (see
// edge_triangles), so the matrix holds twice the coefficients of the other classes
// and yields twice the counts.
void partial_matrix(int k, const int16_t *lut, const uint32_t *class_code, std::vector<uint32_t> &out) {
    const int N = num_classes(k);
    std::vector<int> coef((size_t)N * N, 0);
    for (int c = 0; c < N; c++) {
        const uint32_t code = class_code[c];
        uint32_t edge[10];
        int edges = 0, deg[5] = {};
        for (int i = 0; i < k; i++)
            for (int j = i + 1; j < k; j++) {
                const uint32_t bits = code & ((1u << code_bit(k, i, j)) | (1u << code_bit(k, j, i)));
                if (!bits) continue;
                edge[edges++] = bits;
                deg[i]++;
                deg[j]++;
            }
        bool deg3 = false;
        for (int i = 0; i < k; i++) deg3 = deg3 || deg[i] == 3;
        const int unit = k == 4 && !(edges == 4 && deg3) ? 2 : 1;
        for (uint32_t sub = 0; sub < 1u << edges; sub++) {
            uint32_t kept = 0;
            int left = edges;
            for (int e = 0; e < edges; e++)
                if ((sub >> e) & 1u) {
                    kept |= edge[e];
                    left--;
                }
            const int to = lut[kept];
            if (to >= 0) coef[(size_t)to * N + c] += left & 1 ? -unit : unit;
        }
    }
    out.assign(1, 0u);
    for (int to = 0; to < N; to++)
        for (int c = 0; c < N; c++)
            if (coef[(size_t)to * N + c])
                out.push_back(((uint32_t)to << 24) | ((uint32_t)c << 16) | (uint32_t)(coef[(size_t)to * N + c] + 32768));
    out[0] = (uint32_t)out.size() - 1u;
}

int launch_partial(int k, PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s, int grid_num,
                   int grid_den) {
    int launches = 0;
    if (k == 3) launch_pdl(k_partial_prep<3>, grid_prep(max_entries, num_sms), 256, 0, s, a);
    else launch_pdl(k_partial_prep<4>, grid_prep(max_entries, num_sms), 256, 0, s, a);
    if (!launched()) return ACC_ERR_CUDA;
    launches++;
    if (k == 3) {
        const int g3 = scaled_grid(4, num_sms, grid_num, grid_den);
        if (a.nh) launch_pdl(k_partial3<true>, g3, kPThreads, 0, s, a);
        else launch_pdl(k_partial3<false>, g3, kPThreads, 0, s, a);
        if (!launched()) return ACC_ERR_CUDA;
        launches++;
    } else {
        for (int phase = 1; phase <= 2; phase++) {
            const int rc = wedges<4, false>(a, phase, num_sms, s, grid_num, grid_den);
            if (rc < 0) return rc;
            launches += rc;
        }
    }
    const int fin = finish_grid(a, max_entries, num_sms);
    if (k == 3) launch_pdl(k_partial_finish<3, true>, fin, kFThreads, 0, s, a);
    else launch_pdl(k_partial_finish<4, true>, fin, kFThreads, 0, s, a);
    return launched() ? launches + 1 : ACC_ERR_CUDA;
}

int launch_partial5_prep(const PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s) {
    launch_pdl(k_partial_prep<5>, grid_prep(max_entries, num_sms), 256, 0, s, a);
    return launched() ? 1 : ACC_ERR_CUDA;
}

int launch_partial5_wedges(const PartialArgs &a, int phase, int num_sms, cudaStream_t s, int grid_num, int grid_den) {
    return wedges<4, true>(a, phase, num_sms, s, grid_num, grid_den);
}

int launch_partial5_finish(PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s) {
    const int fin = finish_grid(a, max_entries, num_sms);
    launch_pdl(k_partial_finish<4, false>, fin, kFThreads, 0, s, a);
    return launched() ? 1 : ACC_ERR_CUDA;
}

int launch_partial5_pairs(const PartialArgs &a, int phase, int num_sms, cudaStream_t s, int grid_num, int grid_den) {
    return wedges<5, false>(a, phase, num_sms, s, grid_num, grid_den);
}

}  // namespace acc
