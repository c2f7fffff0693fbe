// Counting by partial patterns, k = 5 (see partial.cu for k = 3, 4 and the
// inclusion and exclusion from partial counts P to induced ones).
//
// The 21 connected graphs on five vertices, typed by the states of their
// edges, are counted as partial patterns:
//   directly, each occurrence a fixed number of times: the star K_{1,4}, the
//     5-cycle, K_{2,3}, K_{1,1,3} (an edge with three common neighbours), and
//     what holds a diamond whose tips have a further common neighbour (a
//     diamond with its tips joined through a vertex, the wheel, K_5 less one or
//     two edges, K_4 with a vertex on one or two of its vertices, K_5);
//   as products of smaller counts in which vertices that the pattern does not
//     join may coincide: the fork, the path, triangles and diamonds with
//     pendants, two triangles on a vertex, banner, house, fan.  The sums with
//     coinciding vertices are those of the quotient patterns on four, three
//     and two vertices, whose partial counts are known; they are taken off at
//     the end (k_quotients), one partition of the five vertices at a time.
// A class's sum is divided by the number of times an occurrence is counted
// (div5: for the products the automorphisms of the undirected pattern).
//
// What is visited: wedges between a pair of vertices (partial.cu, also for the
// houses and banners), 3-paths above a 5-cycle's smallest vertex, triangles,
// and for every diamond the neighbours of one tip.  The list scan (enum.cu)
// instead reads the lists of every connected triple.
#include <string.h>

#include <type_traits>

#include "partial.cuh"

namespace acc {

namespace {

constexpr int kN5 = num_classes(5);


__device__ __forceinline__ Bins5 bins5(const PartialArgs &a, uint32_t *lo) {
    return Bins5{lo, a.p5.sums, a.p5.lut5, a.status};
}

__device__ __forceinline__ PView view5(const PartialArgs &a) { return pview(a, a.gs.one); }

// ---------------------------------------------------------------------------
// Products at a vertex: n (typed degree), q (2-walks from it by their two
// states) and t (triangles at it, ordered, by the states of its two edges and
// of the third).  A block takes 32 vertices at a time: a warp gathers the 39
// sums of four of them from their neighbours, then a thread per product adds
// its term for each.
// ---------------------------------------------------------------------------
// 60000 vertices: 81 us (211 with the stars' binomials on 15 threads and tiles of
// 32 vertices); bound by the gather's loads and, on small graphs, by its few tiles.
constexpr int kVWarps = 8, kVThreads = kVWarps * kWarp, kVTile = 16;
constexpr int kF = 49;  // n[3], q[9], t[27], 1, n choose 2, 3, 4 [3 each]
constexpr int kTreeTerms = 54 + 45 + 15 + 8, kTriTerms = 27 * 6 + 27 * 9 + 378;

// Product o: its code, weight and factors (indexes into the 49 values).  The
// last 8 of the tree terms are counts of smaller patterns: code 2^20 + i for
// entry i of Partial5::small.
__device__ void vertex_term(int o, const int16_t *lut3, uint32_t *code, uint32_t *weight, int *f) {
    // the m-th pair i <= j of x values
    auto pair = [](int m, int x, int *i, int *j) {
        int a = 0;
        while (m >= x - a) {
            m -= x - a;
            a++;
        }
        *i = a;
        *j = a + m;
    };
    // m of the neighbours of state s + 1
    auto choose = [](int s, int m) -> int { return m == 0 ? 39 : (m == 1 ? s : 40 + 3 * (m - 2) + s); };
    f[2] = 39;
    *weight = 1;
    if (o < 54) {  // fork: w1 = y, w2, w3 leaves, w4 beyond y
        const int k = o / 6;
        int i, j;
        pair(o % 6, 3, &i, &j);
        f[0] = i;
        f[1] = j;
        f[2] = 3 + k;
        *code = e5(0, 1, k / 3 + 1) | e5(0, 2, i + 1) | e5(0, 3, j + 1) | e5(1, 4, k % 3 + 1);
        if (i != j) *weight = 2;
        return;
    }
    o -= 54;
    if (o < 45) {  // path: w1, w2 next to the middle, w3, w4 the ends
        int i, j;
        pair(o, 9, &i, &j);
        f[0] = 3 + i;
        f[1] = 3 + j;
        *code = e5(0, 1, i / 3 + 1) | e5(1, 3, i % 3 + 1) | e5(0, 2, j / 3 + 1) | e5(2, 4, j % 3 + 1);
        if (i != j) *weight = 2;
        return;
    }
    o -= 45;
    if (o < 15) {  // star: m1 + m2 + m3 = 4 leaves by state
        int m1 = 0;
        while (o >= 5 - m1) o -= 5 - m1++;
        const int m2 = o, m3 = 4 - m1 - m2;
        f[0] = choose(0, m1);
        f[1] = choose(1, m2);
        f[2] = choose(2, m3);
        auto leaf = [&](int t) -> uint32_t { return t <= m1 ? 1u : (t <= m1 + m2 ? 2u : 3u); };
        *code = e5(0, 1, leaf(1)) | e5(0, 2, leaf(2)) | e5(0, 3, leaf(3)) | e5(0, 4, leaf(4));
        return;
    }
    o -= 15;
    if (o < 8) {  // open triples of k = 3 by the states of their two edges; arcs by state 1 and 3
        int i = 0, j = 0;
        if (o < 6) pair(o, 3, &i, &j);
        f[0] = o < 6 ? (i == j ? choose(i, 2) : i) : (o == 6 ? 0 : 2);
        f[1] = o < 6 && i != j ? j : 39;
        *code = (1u << 20) + (o < 6 ? (uint32_t)__ldg(lut3 + (((i + 1) << 4) | (j + 1))) : 7u + (uint32_t)o);
        return;
    }
    o -= 8;
    auto triangle = [](int t, int y, int z) -> uint32_t {
        return e5(0, y, t / 9 + 1) | e5(0, z, (t / 3) % 3 + 1) | e5(y, z, t % 3 + 1);
    };
    if (o < 27 * 6) {  // two pendants
        int i, j;
        pair(o % 6, 3, &i, &j);
        f[0] = 12 + o / 6;
        f[1] = i;
        f[2] = j;
        *code = triangle(o / 6, 1, 2) | e5(0, 3, i + 1) | e5(0, 4, j + 1);
        if (i != j) *weight = 2;
        return;
    }
    o -= 27 * 6;
    if (o < 27 * 9) {  // a tail of two edges
        const int k = o % 9;
        f[0] = 12 + o / 9;
        f[1] = 3 + k;
        *code = triangle(o / 9, 1, 2) | e5(0, 3, k / 3 + 1) | e5(3, 4, k % 3 + 1);
        return;
    }
    o -= 27 * 9;
    int i, j;  // two triangles
    pair(o, 27, &i, &j);
    f[0] = 12 + i;
    f[1] = 12 + j;
    *code = triangle(i, 1, 2) | triangle(j, 3, 4);
    if (i != j) *weight = 2;
}

__global__ void __launch_bounds__(kVThreads) k_vertex5(PartialArgs a) {
    const JoinsPrevious beside;  // k_wedges<5, 2>
    if (scan_instead(a)) return;
    constexpr int kTerms = kTreeTerms + kTriTerms, kPer = (kTerms + kVThreads - 1) / kVThreads;
    __shared__ unsigned long long F[kVTile][kF];
    __shared__ int closed[kVTile], nclosed;
    const PView g = view5(a);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    uint32_t code[kPer], weight[kPer];
    int f[kPer][3];
    unsigned long long acc[kPer];
#pragma unroll
    for (int i = 0; i < kPer; i++) {
        acc[i] = 0;
        code[i] = weight[i] = 0;
        f[i][0] = f[i][1] = f[i][2] = 39;
        if (threadIdx.x + i * kVThreads < kTerms) vertex_term(threadIdx.x + i * kVThreads, a.p5.lut3, &code[i], &weight[i], f[i]);
    }
    for (int v0 = blockIdx.x * kVTile; v0 < g.n; v0 += gridDim.x * kVTile) {
        if (threadIdx.x == 0) nclosed = 0;
        __syncthreads();
        for (int k = wib; k < kVTile; k += kVWarps) {
            const int x = v0 + k;
            unsigned long long q[9] = {}, tau = 0;  // (tau: lane i holds t[i])
            if (x < g.n) {
                const long long b = g.nptr[x];
                const int d = g.deg[x];
                const bool tri = a.p5.in_tri[x] != 0;
                for (int j0 = 0; j0 < d; j0 += kWarp) {
                    const int j = j0 + lane;
                    uint32_t s = 0;
                    EdgeTri t = {{0ull, 0ull, 0ull}, false};
                    if (j < d) {
                        const uint32_t e = __ldg(a.nbr + b + j);
                        s = e & 3u;
                        const unsigned long long ny = g.nd[e >> 2];
#pragma unroll
                        for (uint32_t i = 0; i < 9; i++) q[i] += s == i / 3u + 1u ? nd_of(ny, i % 3u + 1u) : 0ull;
                        if (tri) t = edge_tri(a, b + j, (int)(e >> 2) > x);
                    }
                    for (unsigned m = __ballot_sync(kFull, t.any()); m; m &= m - 1u) {
                        const int h = __ffs(m) - 1;
                        EdgeTri th;
#pragma unroll
                        for (int i = 0; i < 3; i++) th.w[i] = __shfl_sync(kFull, t.w[i], h);
                        th.flip = __shfl_sync(kFull, (int)t.flip, h) != 0;
                        const uint32_t sh = __shfl_sync(kFull, s, h);
                        // t[9 s(x,y) + 3 s(x,z) + s(y,z)]
                        if (lane < 27 && (uint32_t)lane / 9u + 1u == sh)
                            tau += th.get(((uint32_t)lane / 3u) % 3u, (uint32_t)lane % 3u);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 9; i++) {
#pragma unroll
                for (int d = 16; d; d >>= 1) q[i] += __shfl_xor_sync(kFull, q[i], d);
                if (lane == 0) F[k][3 + i] = q[i];
            }
            const unsigned long long nd = x < g.n ? g.nd[x] : 0ull;
            if (lane < 3) F[k][lane] = nd_of(nd, lane + 1u);
            if (lane < 27) F[k][12 + lane] = tau;
            if (lane == 0) F[k][39] = 1ull;
            if (lane < 9) {
                const unsigned long long n = nd_of(nd, (uint32_t)lane % 3u + 1u);
                const unsigned long long c2 = n > 1 ? n * (n - 1) / 2 : 0ull, c3 = n > 2 ? c2 * (n - 2) / 3 : 0ull;
                F[k][40 + lane] = lane < 3 ? c2 : (lane < 6 ? c3 : (n > 3 ? c3 * (n - 3) / 4 : 0ull));
            }
            if (__ballot_sync(kFull, tau != 0ull) && lane == 0) closed[atomicAdd(&nclosed, 1)] = k;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const int o = threadIdx.x + i * kVThreads;
            if (o < kTreeTerms) {
                for (int k = 0; k < kVTile; k++) acc[i] += F[k][f[i][0]] * F[k][f[i][1]] * F[k][f[i][2]];
            } else if (o < kTerms) {
                for (int c = 0; c < nclosed; c++) {
                    const unsigned long long *x = F[closed[c]];
                    acc[i] += x[f[i][0]] * x[f[i][1]] * x[f[i][2]];
                }
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < kPer; i++) {
        const unsigned long long x = acc[i] * weight[i];
        if (!x) continue;
        if (code[i] >> 20) {
            atomicAdd(&a.p5.small[code[i] & 31u], x);
            continue;
        }
        const int cls = (int)__ldg(a.p5.lut5 + code[i]);
        if (cls < 0) set_status(a.status, ACC_ERR_INTERNAL);
        else atomicAdd(&a.p5.sums[cls], x);
    }
}

// ---------------------------------------------------------------------------
// Products at an edge with common neighbours and at a triangle.
// ---------------------------------------------------------------------------

// Thread per edge (upper entry), and per triangle corner below: 27 us on 866
// triangles, 88 on 16000 (157 with a thread per triangle over all type pairs, not
// only the nonzero ones); bound by the chains of class lookups and adds.
// On an edge: triangles on it with a pendant at both ends
// (twice: the ends may be swapped), two of them with a pendant at one end, and
// three of them.
__device__ void edge_sums(const PartialArgs &a, const PView &g, const Bins5 &bins, long long pos) {
    const uint32_t r = a.src[pos];
    if (r >> 31) return;
    const EdgeTri t = edge_tri(a, pos, true);
    const uint32_t types = types_of(t);
    if (!types) return;
    const uint32_t e = a.nbr[pos], s = e5(0, 1, e & 3u);
    const unsigned long long nx = g.nd[r], ny = g.nd[e >> 2];
    auto page = [](int m, uint32_t z) -> uint32_t { return e5(0, m, z / 3u + 1u) | e5(1, m, z % 3u + 1u); };
    for (uint32_t mz = types; mz; mz &= mz - 1u) {
        const uint32_t z = next_bit(mz);
        const unsigned long long c = t.get(z / 3u, z % 3u);
        for (uint32_t i = 1; i <= 3; i++)
            for (uint32_t j = 1; j <= 3; j++) {
                const unsigned long long x = nd_of(nx, i) * nd_of(ny, j);
                if (x) bins.add(s | page(2, z) | e5(0, 3, i) | e5(1, 4, j), 2u * c * x);
            }
        for (uint32_t my = mz; my; my &= my - 1u) {
            const uint32_t y = next_bit(my);
            const unsigned long long d = t.get(y / 3u, y % 3u);
            // two common neighbours in either order (they may coincide)
            const unsigned long long two = y == z ? c * c : 2u * c * d;
            for (uint32_t i = 1; i <= 3; i++) {
                const unsigned long long px = nd_of(nx, i), py = nd_of(ny, i);
                if (px) bins.add(s | page(2, z) | page(3, y) | e5(0, 4, i), two * px);
                if (py) bins.add(s | page(2, z) | page(3, y) | e5(1, 4, i), two * py);
            }
            // three different ones
            const unsigned long long pairs = y == z ? c * (c - 1u) / 2 : c * d;
            for (uint32_t mx = my; mx; mx &= mx - 1u) {
                const uint32_t x = next_bit(mx);
                const unsigned long long b = t.get(x / 3u, x % 3u);
                unsigned long long n;
                if (x == y) n = y == z ? (c > 2 ? c * (c - 1u) / 2 * (c - 2u) / 3 : 0ull) : c * (d * (d - 1u) / 2);
                else n = pairs * b;
                if (n) bins.add(s | page(2, z) | page(3, y) | page(4, x), n);
            }
        }
    }
}

// Thread per corner c of a triangle v < u < w (x, y its other two vertices):
// diamonds with spine x, y, tip c and a pendant at c (twice: the spine may be
// swapped); fans with hub c and middle x, y (twice: the path may be turned
// round); the 5-cycle pass's walks that pass c twice (below).
__device__ void corner_sums(const PartialArgs &a, const PView &g, const Bins5 &bins, unsigned long long i, uint32_t k) {
    const uint4 tr = a.p5.tris[i];
    const uint32_t pvu = tr.x, puw = tr.y, pvw = tr.z;
    const uint32_t v = a.src[pvu] & 0x7FFFFFFFu, evu = a.nbr[pvu], euw = a.nbr[puw], evw = a.nbr[pvw];
    const uint32_t u = evu >> 2, w = euw >> 2, svu = evu & 3u, suw = euw & 3u, svw = evw & 3u;
    if (k == 0u) {
        const int c3 = (int)__ldg(a.p5.lut3 + ((svu << 4) | svw | (suw << 2)));
        if (c3 >= 0) atomicAdd(&a.p5.small[c3], 1ull);
    }
    const uint32_t c = k == 0u ? v : (k == 1u ? u : w);
    const uint32_t sxy = k == 0u ? suw : (k == 1u ? svw : svu);
    const uint32_t scx = k == 0u ? svu : (k == 1u ? swap_state(svu) : swap_state(svw));
    const uint32_t scy = k == 0u ? svw : (k == 1u ? suw : swap_state(suw));
    const EdgeTri xy = edge_tri(a, k == 0u ? puw : (k == 1u ? pvw : pvu), true);
    EdgeTri cx = edge_tri(a, k == 2u ? pvw : pvu, true), cy = edge_tri(a, k == 0u ? pvw : puw, true);
    cx.flip = k != 0u;
    cy.flip = k == 2u;
    // neighbours of c below v
    const int lower = k == 0u ? g.lo[v]
                              : (int)((long long)a.rev[k == 1u ? pvu : pvw].x - 1 - g.nptr[c]);
    const uint32_t d0 = e5(0, 1, sxy) | e5(0, 2, swap_state(scx)) | e5(1, 2, swap_state(scy));
    const unsigned long long nc = g.nd[c];
    for (uint32_t m = types_of(xy); m; m &= m - 1u) {
        const uint32_t z = next_bit(m);
        const unsigned long long n = xy.get(z / 3u, z % 3u);
        for (uint32_t s = 1; s <= 3; s++) {
            const unsigned long long p = nd_of(nc, s);
            if (p) bins.add(d0 | e5(0, 3, z / 3u + 1u) | e5(1, 3, z % 3u + 1u) | e5(2, 4, s), 2u * n * p);
        }
    }
    // fan: hub c (w0), middle x, y (w1, w2), ends w3 at c, x and w4 at c, y
    const uint32_t f0 = e5(0, 1, scx) | e5(0, 2, scy) | e5(1, 2, sxy), my = types_of(cy);
    for (uint32_t m = types_of(cx); m; m &= m - 1u) {
        const uint32_t z = next_bit(m);
        const unsigned long long n = cx.get(z / 3u, z % 3u);
        for (uint32_t r = my; r; r &= r - 1u) {
            const uint32_t q = next_bit(r);
            bins.add(f0 | e5(0, 3, z / 3u + 1u) | e5(1, 3, z % 3u + 1u) | e5(0, 4, q / 3u + 1u) | e5(2, 4, q % 3u + 1u),
                     2u * n * cy.get(q / 3u, q % 3u));
        }
    }
    // walks r - c - x - y - c - r from r below the whole triangle: the 5-cycle
    // pass counts them with both its neighbours of r being c
    unsigned long long below = 0;
    const long long cb = g.nptr[c];
#pragma unroll 4
    for (int j = 0; j < lower; j++) below += 1ull << (kNdBits * ((__ldg(a.nbr + cb + j) & 3u) - 1u));
    for (uint32_t s = 1; s <= 3; s++) {
        const unsigned long long n = nd_of(below, s);
        const uint32_t src = swap_state(s);  // state(r, c)
        if (n)
            bins.add(e5(0, 1, src) | e5(1, 2, scx) | e5(2, 3, sxy) | e5(3, 4, swap_state(scy)) | e5(0, 4, src), 0ull - n);
    }
}

__global__ void __launch_bounds__(256) k_closed5(PartialArgs a) {
    const JoinsPrevious beside;  // k_wedges<5, 2>
    const unsigned long long tris = a.p5.ctr[kCtrTris];
    if (!tris) return;
    __shared__ int instead;
    ask_scan(a, &instead);
    extern __shared__ __align__(16) unsigned char smem[];
    const Bins5 bins = bins5(a, reinterpret_cast<uint32_t *>(smem));
    bins.clear();
    if (instead) return;
    const PView g = view5(a);
    // (thread t of block b takes item t gridDim + b: few items still reach every SM)
    const long long t0 = threadIdx.x * (long long)gridDim.x + blockIdx.x, step = (long long)gridDim.x * blockDim.x;
    for (long long i = t0; i < 3 * (long long)tris; i += step)
        corner_sums(a, g, bins, (unsigned long long)(i / 3), (uint32_t)(i % 3));
    const long long nnz = a.info->nnz;
    for (long long p = t0; p < nnz; p += step)
        if (a.p5.in_tri[a.src[p] & 0x7FFFFFFFu]) edge_sums(a, g, bins, p);
    bins.flush();
}

// ---------------------------------------------------------------------------
// Diamonds.  A warp takes a triangle's edge as the spine x < y and its third
// vertex a as a tip, finds the other tips b > a among the neighbours of y
// (adjacent to x too), and for each reads the neighbours z of b adjacent to a:
// with them everything that holds the diamond and a vertex on both tips.  208 us
// for 1.9e5 diamonds (1899 vertices, 20296 arcs), 18 us for 1600: the reads of the
// tips' lists and two to four states an entry, from L2.
// ---------------------------------------------------------------------------
template <bool HASH>
__global__ void __launch_bounds__(256, 2) k_diamonds5(PartialArgs a) {
    const JoinsPrevious beside;  // k_wedges<5, 2>
    const unsigned long long units = 3ull * a.p5.ctr[kCtrTris];
    if (!units) return;
    __shared__ int instead;
    ask_scan(a, &instead);
    extern __shared__ __align__(16) unsigned char smem[];
    const Bins5 bins = bins5(a, reinterpret_cast<uint32_t *>(smem));
    bins.clear();
    if (instead) return;
    const PView g = view5(a);
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned long long un = 0;
        if (lane == 0) un = atomicAdd(&a.p5.ctr[kCtrDiamond], 1ull);
        un = __shfl_sync(kFull, un, 0);
        if (un >= units) break;
        const uint4 tr = a.p5.tris[un / 3u];
        const uint32_t k = (uint32_t)(un % 3u);
        const uint32_t v = a.src[tr.x] & 0x7FFFFFFFu, evu = a.nbr[tr.x], euw = a.nbr[tr.y], evw = a.nbr[tr.z];
        const uint32_t u = evu >> 2, w = euw >> 2, svu = evu & 3u, suw = euw & 3u, svw = evw & 3u;
        const uint32_t x = k == 2u ? u : v, y = k == 0u ? u : w, t = k == 0u ? w : (k == 1u ? u : v);
        const uint32_t sxy = k == 0u ? svu : (k == 1u ? svw : suw);
        const uint32_t sxt = k == 0u ? svw : (k == 1u ? svu : swap_state(svu));
        const uint32_t syt = k == 0u ? suw : (k == 1u ? swap_state(suw) : swap_state(svw));
        const uint32_t base = e5(0, 1, sxy) | e5(0, 2, sxt) | e5(1, 2, syt);
        const long long yb = g.nptr[y];
        const int yd = g.deg[y];
        for (int j0 = lower_id(a.nbr + yb, yd, t + 1u); j0 < yd; j0 += kWarp) {
            uint32_t b = 0, off = 0, code = 0, sab = 0;
            int len = 0;
            if (j0 + lane < yd) {
                const uint32_t e = __ldg(a.nbr + yb + j0 + lane);
                const uint32_t sxb = e >> 2 == x ? 0u : pstate<HASH>(g, x, e >> 2);
                if (sxb) {
                    b = e >> 2;
                    code = base | e5(0, 3, sxb) | e5(1, 3, e & 3u);
                    off = (uint32_t)g.nptr[b];
                    len = g.deg[b];
                    sab = pstate<HASH>(g, t, b);
                    if (sab && y < t) {  // x < y < t < b: each K_4 once, with a pendant at each vertex
                        const uint32_t c4 = code | e5(2, 3, sab);
                        const unsigned long long n[4] = {g.nd[x], g.nd[y], g.nd[t], g.nd[b]};
                        const uint32_t sv[6] = {sxy, sxt, sxb, syt, e & 3u, sab};  // 01 02 03 12 13 23
                        for (int i = 0; i < 4; i++)
                            for (uint32_t s = 1; s <= 3; s++) {
                                unsigned long long p = nd_of(n[i], s);
                                int m = 0;
                                for (int r = 0; r < 4; r++)
                                    for (int q = r + 1; q < 4; q++, m++) {
                                        if (r == i && sv[m] == s) p--;
                                        if (q == i && swap_state(sv[m]) == s) p--;
                                    }
                                if (p) bins.add(c4 | (s << (2 * i)), p);  // (field of slot 4 is the lowest)
                            }
                    }
                }
            }
            int tot;
            const int pre = warp_excl(len, lane, &tot);
            off -= (uint32_t)pre;
            for (int f0 = 0; f0 < tot; f0 += kWarp) {
                const int f = f0 + lane;
                int r = 0;  // the last tip whose list starts at or before f
#pragma unroll
                for (int d = 16; d; d >>= 1)
                    if (__shfl_sync(kFull, pre, r + d) <= f) r += d;
                const uint32_t hb = __shfl_sync(kFull, b, r), ho = __shfl_sync(kFull, off, r);
                const uint32_t hc = __shfl_sync(kFull, code, r), hs = __shfl_sync(kFull, sab, r);
                if (f < tot) {
                    const uint32_t e = __ldg(a.nbr + (ho + (uint32_t)f)), z = e >> 2;
                    const uint32_t stz = z == x || z == y || z == t ? 0u : pstate<HASH>(g, t, z);
                    if (stz) {
                        const uint32_t on = hc | e5(2, 4, stz) | e5(3, 4, e & 3u);
                        const uint32_t sxz = pstate<HASH>(g, x, z), syz = pstate<HASH>(g, y, z);
                        bins.add(on, 1ull);                                     // tips joined through z
                        if (hs) bins.add(on | e5(2, 3, hs), 1ull);              // K_4 and z on two of its vertices
                        if (sxz) bins.add(on | e5(0, 4, sxz), 1ull);            // wheels with hub x, y
                        if (syz) bins.add(on | e5(1, 4, syz), 1ull);
                        if (sxz && syz) {
                            bins.add(on | e5(0, 4, sxz) | e5(1, 4, syz), 1ull);  // triangle x, y, z and two tips
                            if (hs && y < t && z > hb)                           // x < y < t < b < z: each K_5 once
                                bins.add(on | e5(0, 4, sxz) | e5(1, 4, syz) | e5(2, 3, hs), 1ull);
                        }
                    }
                }
            }
        }
    }
    bins.flush();
}

// ---------------------------------------------------------------------------
// 5-cycles, from their smallest vertex c: the wedges c - b - x above c by
// their end x (a table, as in partial.cu, with the state of c and x in the
// first word's top bits), then for every edge x - y between two ends the pairs
// of a wedge to x and a wedge to y.  Wedges through the other end are left out
// there; pairs through one vertex are taken off by corner_sums.  Bound by the
// latency of the list entries and table lookups; roots with up to 128 wedges take
// a warp, the others a block (60000 vertices: 116 + 214 us; with 25 roots a grab
// phase 1 took 1809, with two searched ranges for every root phase 2 took 372).
// ---------------------------------------------------------------------------
constexpr int kCWarps = 8, kCThreads = kCWarps * kWarp;
#ifndef ACC_CYCLE_SLOTS
#define ACC_CYCLE_SLOTS 4096
#endif
// Tables: one a warp for the roots with few wedges (three blocks an SM), one a
// block for the others (two).
constexpr int kLSlots = 192, kLFill = kLSlots * 2 / 3, kLRoots = 16;
constexpr int kCSlots = ACC_CYCLE_SLOTS, kCFill = kCSlots * 2 / 3;
static_assert(kLSlots >= 96 && kCSlots >= 96, "a probe steps at most 91 slots");
constexpr int kCParts = 16;     // most blocks a root's range pairs are dealt to
constexpr int kCRows = 64, kCRing = 4 * kCRows;
constexpr int kCRanges = 512;   // end ranges of one root

struct CycleTable {
    uint32_t *t;  // (key, three words of three 10-bit counts), key = (root - first root + 1) << 26 | end
    uint32_t slots;
    __device__ __forceinline__ int at(uint32_t key, bool insert) const {
        const uint32_t h = key * 0x9E3779B1u;
        uint32_t i = (uint32_t)(((unsigned long long)h * slots) >> 32);
        const uint32_t step = 6u * ((h >> 4) & 15u) + 1u;
        for (uint32_t tries = 0; tries < slots; tries++, i = i + step < slots ? i + step : i + step - slots) {
            const uint32_t old = insert ? atomicCAS(&t[4 * i], 0u, key) : t[4 * i];
            if (old == key || (insert && !old)) return (int)i;
            if (!old) return -1;
        }
        return -1;
    }
};

// Rows [0, nrows) as one flat sequence, an entry a lane (the whole warp):
// row(j, &first, pay) gives row j's part of the lists nbr, entry(e, pay) takes
// an entry; two windows of 32 entries are in flight.
template <typename Row, typename Entry>
__device__ __forceinline__ unsigned flat_rows(const uint32_t *__restrict__ nbr, uint32_t *ring, int lane, int nrows,
                                              Row row, Entry entry) {
    constexpr int RM = kCRows - 1;
    constexpr int W = 2;
    uint32_t *rS = ring, *rO = ring + kCRows, *rP = ring + 2 * kCRows, *rQ = ring + 3 * kCRows;
    uint32_t T = 0, F = 0;
    int tail = 0, cur = -1, jb = 0;
    for (;;) {
        while (jb < nrows && T - F < 32u * W && tail - cur + kWarp <= kCRows) {
            uint32_t first = 0;
            uint2 pay = make_uint2(0u, 0u);
            const int cnt = jb + lane < nrows ? row(jb + lane, &first, &pay) : 0;
            const unsigned nz = __ballot_sync(kFull, cnt > 0);
            jb += kWarp;
            if (!nz) continue;
            int tot;
            const int pre = warp_excl(cnt, lane, &tot);
            if (cnt > 0) {
                const int slot = (tail + __popc(nz & ((1u << lane) - 1u))) & RM;
                rS[slot] = T + (uint32_t)pre;
                rO[slot] = first - (T + (uint32_t)pre);
                rP[slot] = pay.x;
                rQ[slot] = pay.y;
            }
            tail += __popc(nz);
            T += (uint32_t)tot;
        }
        const uint32_t pend = T - F;
        if (!pend) break;
        __syncwarp();
        uint32_t e[W], pos[W];
        uint2 pay[W];
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
            const int at = (cur + __popc(starts & (0xFFFFFFFFu >> (31 - lane)))) & RM;
            cur += __popc(starts);
            pos[w] = rO[at] + t0 + (uint32_t)lane;
            pay[w] = make_uint2(rP[at], rQ[at]);
            e[w] = 32u * w + (uint32_t)lane < pend ? __ldg(nbr + pos[w]) : 0u;
        }
#pragma unroll
        for (int w = 0; w < W; w++)
            if (32u * w + (uint32_t)lane < pend) entry(e[w], pay[w]);
        F += pend < 32u * W ? pend : 32u * W;
    }
    __syncwarp();
    return T;
}

// What one warp does of a table pass: rows of the roots' upper entries p0, p0 +
// step, ... (roots v0, v0 + 1, ...), ends in [lo, hi) or [lo2, hi2).
struct CycleWarp {
    const PartialArgs *a;
    PView g;
    CycleTable tab;
    Bins5 bins;
    uint32_t *ring;
    int lane;

    __device__ __forceinline__ int part(long long p, uint32_t lo, uint32_t hi, bool all, uint32_t *first) const {
        const uint2 r = __ldg(a->rev + p);
        *first = r.x;
        return all || !r.y ? (int)r.y : id_range(a->nbr, (int)r.y, lo, hi, first);
    }
    __device__ __forceinline__ void fill(long long p0, long long step, int nrows, uint32_t v0, uint32_t lo, uint32_t hi,
                                         bool all) {
        flat_rows(a->nbr, ring, lane, nrows,
            [&](int j, uint32_t *first, uint2 *pay) -> int {
                const long long p = p0 + (long long)j * step;
                const uint32_t r = __ldg(a->src + p);
                if (r >> 31) return 0;
                *pay = make_uint2(__ldg(a->nbr + p), (r - v0 + 1u) << 26);
                return part(p, lo, hi, all, first);
            },
            [&](uint32_t e, uint2 pay) {
                const int i = tab.at(pay.y | (e >> 2), true);
                if (i < 0) set_status(a->status, ACC_ERR_INTERNAL);
                else atomicAdd(&tab.t[4 * i + (pay.x & 3u)], 1u << (10 * ((e & 3u) - 1u)));
            });
    }
    // states of the root to its neighbours that are ends
    __device__ __forceinline__ void mark(long long p0, long long step, int nrows, uint32_t v0) {
        for (int j = lane; j < nrows; j += kWarp) {
            const long long p = p0 + (long long)j * step;
            const uint32_t r = __ldg(a->src + p);
            if (r >> 31) continue;
            const uint32_t e = __ldg(a->nbr + p);
            const int i = tab.at(((r - v0 + 1u) << 26) | (e >> 2), false);
            if (i >= 0) atomicOr(&tab.t[4 * i + 1], (e & 3u) << 30);
        }
        __syncwarp();
    }
    // edges x - y, x in [lo, hi), y > x in [lo2, hi2), both ends of one root,
    // x's slots s0, s0 + step, ...
    __device__ __forceinline__ void edges(int s0, int step, uint32_t lo, uint32_t hi, uint32_t lo2, uint32_t hi2) {
        const int n = s0 < (int)tab.slots ? ((int)tab.slots - s0 + step - 1) / step : 0;
        flat_rows(a->nbr, ring, lane, n,
            [&](int j, uint32_t *first, uint2 *pay) -> int {
                const uint32_t slot = (uint32_t)(s0 + j * step), key = tab.t[4 * slot], x = key & 0x3FFFFFFu;
                if (!key || x < lo || x >= hi) return 0;
                *pay = make_uint2(slot, key);
                const int l = g.lo[x];
                *first = (uint32_t)(g.nptr[x] + l);
                return g.deg[x] - l;
            },
            [&](uint32_t e, uint2 pay) {
                const uint32_t y = e >> 2, sxy = e & 3u;
                if (y < lo2 || y >= hi2) return;
                const int i = (int)pay.x, j = tab.at((pay.y & ~0x3FFFFFFu) | y, false);
                if (j < 0) return;
                uint32_t ci[3] = {tab.t[4 * i + 1], tab.t[4 * i + 2], tab.t[4 * i + 3]},
                         cj[3] = {tab.t[4 * j + 1], tab.t[4 * j + 2], tab.t[4 * j + 3]};
                const uint32_t scx = ci[0] >> 30, scy = cj[0] >> 30;
                ci[0] &= 0x3FFFFFFFu;
                cj[0] &= 0x3FFFFFFFu;
                // without the wedge to x through y, and to y through x
#pragma unroll
                for (uint32_t m = 0; m < 3; m++) {
                    if (scy == m + 1u) ci[m] -= 1u << (10 * (swap_state(sxy) - 1u));
                    if (scx == m + 1u) cj[m] -= 1u << (10 * (sxy - 1u));
                }
                const uint32_t mj = types(cj);
                for (uint32_t m = types(ci); m; m &= m - 1u) {
                    const uint32_t z = next_bit(m);
                    const uint32_t code = e5(0, 1, z / 3u + 1u) | e5(1, 2, z % 3u + 1u) | e5(2, 3, sxy);
                    const unsigned long long c = field(ci, z);
                    for (uint32_t r = mj; r; r &= r - 1u) {
                        const uint32_t q = next_bit(r);
                        bins.add(code | e5(0, 4, q / 3u + 1u) | e5(3, 4, swap_state(q % 3u + 1u)), c * field(cj, q));
                    }
                }
            });
    }
    static __device__ __forceinline__ uint32_t field(const uint32_t *c, uint32_t t) {
        return ((t < 3u ? c[0] : (t < 6u ? c[1] : c[2])) >> (10 * (t % 3u))) & 1023u;
    }
    static __device__ __forceinline__ uint32_t types(const uint32_t *c) {
        uint32_t m = 0;
#pragma unroll
        for (int i = 0; i < 3; i++)
#pragma unroll
            for (int j = 0; j < 3; j++) m |= (c[i] >> (10 * j)) & 1023u ? 1u << (3 * i + j) : 0u;
        return m;
    }
};

template <int PHASE>
__global__ void __launch_bounds__(kCThreads, PHASE == 1 ? 3 : 2) k_cycles5(PartialArgs a) {
    grid_dep_wait();
    grid_dep_launch();  // k_wedges<4, PHASE> runs beside
    __shared__ int instead;
    ask_scan(a, &instead);
    unsigned long long *ctr = a.p5.ctr;
    // (the second half of the queue: k_wedges<4> has the first)
    const unsigned long long cap = a.queue_cap / 2;
    uint4 *queue = a.queue + cap;
    if (PHASE == 2 && ctr[kCtrCycTail] == 0) return;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint4 item;
    __shared__ unsigned long long sizes[kCWarps];
    __shared__ uint32_t range[kCRanges + 1];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    constexpr int kTable = PHASE == 1 ? kCWarps * kLSlots : kCSlots;
    uint32_t *table = reinterpret_cast<uint32_t *>(smem), *rings = table + 4 * kTable;
    CycleWarp cw;
    cw.a = &a;
    cw.g = view5(a);
    cw.bins = bins5(a, rings + kCWarps * kCRing);
    cw.ring = rings + wib * kCRing;
    cw.lane = lane;
    cw.tab = CycleTable{PHASE == 1 ? table + 4 * kLSlots * wib : table, (uint32_t)kLSlots};
    for (int i = threadIdx.x; i < 4 * kTable; i += kCThreads) table[i] = 0u;
    cw.bins.clear();
    if (instead) return;  // (after the clear's barrier)
    const PView &g = cw.g;
    if constexpr (PHASE == 1) {
        const long long warps = 4ll * gridDim.x * kCWarps;  // (grabs as in k_wedges)
        const int grab = (int)min(max((long long)(g.n + warps - 1) / warps, 1ll), (long long)kWarp);
        for (;;) {
            unsigned long long u0 = 0;
            if (lane == 0) u0 = atomicAdd(&ctr[kCtrCycUnit], (unsigned long long)grab);
            u0 = __shfl_sync(kFull, u0, 0);
            if ((long long)u0 >= g.n) break;
            const int vl = (int)u0 + lane;
            uint32_t W = 0;
            if (lane < grab && vl < g.n) W = a.p5.cycle_wedges[vl];
            const bool big = W > (uint32_t)kLFill;
            const unsigned heavy = __ballot_sync(kFull, big);
            if (big) {
                // (a table takes one range of ends, or two of half its size)
                const uint32_t r = W <= (uint32_t)kCFill ? 1u : min(W / (uint32_t)(kCFill / 2) + 1u, 5u);
                const uint32_t parts = min(r * (r + 1u) / 2u, (uint32_t)kCParts);
                const unsigned long long i = atomicAdd(&ctr[kCtrCycTail], (unsigned long long)parts);
                if (i + parts > cap) ctr[kCtrScan] = 1ull;
                for (uint32_t c = 0; c < parts && i + c < cap; c++)
                    queue[i + c] = make_uint4((uint32_t)vl, W, c, parts);
            }
            unsigned todo = __ballot_sync(kFull, W > 0u) & ~heavy;
            while (todo) {
                const int s = __ffs(todo) - 1;
                const unsigned after = heavy & ~((1u << s) - 1u);
                const int lim = min(after ? __ffs(after) - 1 : kWarp, s + kLRoots);
                const bool in = ((todo >> lane) & 1u) && lane < lim;
                int tot;
                const int pre = warp_excl(in ? (int)W : 0, lane, &tot);
                const bool ok = in && pre + (int)W <= kLFill;
                const unsigned take = __ballot_sync(kFull, ok);
                const int e = __reduce_max_sync(kFull, ok ? lane : 0);
                const uint32_t v0 = (uint32_t)u0 + s, v1 = (uint32_t)u0 + e;
                const long long p0 = g.nptr[v0] + g.lo[v0], p1 = g.nptr[v1] + g.deg[v1];
                cw.fill(p0, 1, (int)(p1 - p0), v0, 0u, 0u, true);
                cw.mark(p0, 1, (int)(p1 - p0), v0);
                cw.edges(0, 1, 0u, 0x4000000u, 0u, 0x4000000u);
                for (int i = lane; i < kLSlots; i += kWarp)
                    reinterpret_cast<uint4 *>(cw.tab.t)[i] = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
                todo &= ~take;
            }
        }
    } else {
        const unsigned long long tail = min(ctr[kCtrCycTail], cap);
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) {
                const unsigned long long i = atomicAdd(&ctr[kCtrCycHead], 1ull);
                item = i < tail ? queue[i] : make_uint4(0u, 0u, 0u, 0u);
            }
            __syncthreads();
            const uint4 it = item;
            if (!it.y) break;
            const uint32_t v = it.x, n = (uint32_t)g.n;
            const long long pb = g.nptr[v] + g.lo[v];
            const int rows = g.deg[v] - g.lo[v];
            auto size = [&](uint32_t lo, uint32_t hi) -> unsigned long long {
                unsigned long long S = 0;
                for (int r = threadIdx.x; r < rows; r += kCThreads) {
                    uint32_t first;
                    S += (unsigned long long)cw.part(pb + r, lo, hi, false, &first);
                }
#pragma unroll
                for (int d = 16; d; d >>= 1) S += __shfl_xor_sync(kFull, S, d);
                __syncthreads();
                if (lane == 0) sizes[wib] = S;
                __syncthreads();
                S = 0;
                for (int w = 0; w < kCWarps; w++) S += sizes[w];
                return S < (unsigned long long)(hi - lo) ? S : (unsigned long long)(hi - lo);
            };
            // ranges of ends: one that fits the table, or several that fit half of it
            int nr = 0;
            const bool one = it.y <= (uint32_t)kCFill;
            if (one) {
                nr = 1;
            } else {
                uint32_t lo = v + 1u, end = n;
                while (lo < n && nr < kCRanges) {
                    const uint32_t width = end - lo;
                    if (size(lo, end) > (unsigned long long)(kCFill / 2)) {
                        end = lo + width / 2;
                        continue;
                    }
                    if (threadIdx.x == 0) {
                        range[nr] = lo;
                        range[nr + 1] = end;
                    }
                    nr++;
                    lo = end;
                    end = n - lo > 2u * width ? lo + 2u * width : n;
                }
                if (lo < n) {  // (more ranges than kept here)
                    if (threadIdx.x == 0) ctr[kCtrScan] = 1ull;
                    nr = 0;
                }
            }
            __syncthreads();
            const long long p0 = pb + wib;
            const int rw = rows > wib ? (rows - wib + kCWarps - 1) / kCWarps : 0;
            uint32_t sl = one ? 192u : (uint32_t)kCSlots;
            while (one && 2u * sl < 3u * it.y) sl = sl % 3u ? sl + sl / 2u : sl / 3u * 4u;
            cw.tab.slots = sl;
            uint32_t pair = 0;
            for (int i = 0; i < nr; i++)
                for (int j = i; j < nr; j++, pair++) {
                    if (pair % it.w != it.z) continue;
                    const uint32_t lo = one ? v + 1u : range[i], hi = one ? n : range[i + 1], lo2 = one ? lo : range[j],
                                   hi2 = one ? hi : range[j + 1];
                    cw.fill(p0, kCWarps, rw, v, lo, hi, one);
                    if (j > i) cw.fill(p0, kCWarps, rw, v, lo2, hi2, false);
                    __syncthreads();
                    cw.mark(p0, kCWarps, rw, v);
                    __syncthreads();
                    cw.edges(wib, kCWarps, lo, hi, lo2, hi2);
                    __syncthreads();
                    for (uint32_t s = threadIdx.x; s < sl; s += kCThreads)
                        reinterpret_cast<uint4 *>(table)[s] = make_uint4(0u, 0u, 0u, 0u);
                    __syncthreads();
                }
        }
    }
    cw.bins.flush();
}
constexpr size_t cycle_smem(int phase) {
    return 4 * (4 * (phase == 1 ? kCWarps * kLSlots : kCSlots) + kCWarps * kCRing + kN5);
}

// ---------------------------------------------------------------------------
// The quotients, and the counts.
// ---------------------------------------------------------------------------

// Patterns whose sums hold coinciding vertices: their edges as in the sums'
// codes above, and the pairs of vertices that may coincide.
struct Shape {
    int ne;
    unsigned char e[7][2];
    bool apart;  // vertices 0, 2 and 1, 3 are kept apart
};
constexpr int kShapes = 11;
__device__ __forceinline__ Shape shape_of(int s) {
    switch (s) {
    case 0: return {4, {{0, 1}, {0, 2}, {0, 3}, {1, 4}}, false};                                  // fork
    case 1: return {4, {{0, 1}, {1, 3}, {0, 2}, {2, 4}}, false};                                  // path
    case 2: return {5, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {0, 4}}, false};                          // triangle, two pendants at one vertex
    case 3: return {5, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {3, 4}}, false};                          // triangle, tail
    case 4: return {5, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {1, 4}}, false};                          // triangle, pendants at two vertices
    case 5: return {5, {{0, 1}, {1, 2}, {0, 3}, {2, 3}, {0, 4}}, true};                       // 4-cycle, pendant
    case 6: return {6, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {0, 4}, {3, 4}}, false};                  // two triangles
    case 7: return {6, {{0, 1}, {1, 2}, {0, 3}, {2, 3}, {0, 4}, {1, 4}}, true};               // house
    case 8: return {6, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {1, 3}, {2, 4}}, false};                  // diamond, pendant at a tip
    case 9: return {6, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {1, 3}, {0, 4}}, false};                  // diamond, pendant on the spine
    default: return {7, {{0, 1}, {0, 2}, {1, 2}, {0, 3}, {1, 3}, {0, 4}, {2, 4}}, false};         // fan
    }
}
constexpr int kSigma = 81 * 2 + 243 * 4 + 729 * 4 + 2187;
constexpr int kParts = 51;  // partitions of five vertices that join some

// Block of each vertex (three bits a vertex) of partition i.
__device__ __forceinline__ uint32_t partition_of(int i) {
    static constexpr unsigned short part[kParts] = {
        0, 4096, 512, 4608, 8704, 64, 4160, 8256, 576, 4672, 8768, 1088, 5184, 9280, 13376, 8, 4104, 8200,
        520, 4616, 8712, 1032, 5128, 9224, 13320, 72, 4168, 8264, 584, 4680, 8776, 1096, 5192, 9288, 13384,
        136, 4232, 8328, 12424, 648, 4744, 8840, 12936, 1160, 5256, 9352, 13448, 1672, 5768, 9864, 13960};
    return part[i];
}

// Thread per (pattern, states, partition of its vertices): the sum counts the
// maps that join the partition's vertices, as many as the injective maps of
// the quotient pattern: automorphisms times its partial count.  17 us (64 with the
// partitions decoded by a loop).
__global__ void k_quotients(PartialArgs a) {
    grid_dep_wait();
    if (scan_flag(a)) return;  // (no pass that may raise it is left, and no barrier follows)
    // the scan's kernels, launched next, find no unit left
    if (blockIdx.x == 0 && threadIdx.x == 0) a.info->unit_ctr = 1ull << 62;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kSigma * kParts; i += gridDim.x * blockDim.x) {
        int part = i % kParts, sig = i / kParts, sh = 0;
        constexpr int sizes[kShapes] = {81, 81, 243, 243, 243, 243, 729, 729, 729, 729, 2187};
        while (sig >= sizes[sh]) sig -= sizes[sh++];
        const Shape S = shape_of(sh);
        int b[5], nb = 0;
        const uint32_t blocks = partition_of(part);
#pragma unroll
        for (int j = 0; j < 5; j++) {
            b[j] = (int)((blocks >> (3 * j)) & 7u);
            nb = b[j] + 1 > nb ? b[j] + 1 : nb;
        }
        bool ok = true;
        if (S.apart) ok = b[0] != b[2] && b[1] != b[3];
        // states of the quotient's pairs (from its smaller to its larger block)
        uint32_t st[5][5] = {};
        uint32_t code5 = 0;
        int rest = sig;
        for (int e = 0; e < S.ne; e++) {
            const uint32_t s = (uint32_t)(rest % 3) + 1u;
            rest /= 3;
            const int x = S.e[e][0], y = S.e[e][1];
            code5 |= s << ((y == 1 ? 18 : y == 2 ? 14 : y == 3 ? 8 : 0) + 2 * x);
            const int bx = b[x], by = b[y];
            if (bx == by) {
                ok = false;
                continue;
            }
            const int p = bx < by ? bx : by, q = bx < by ? by : bx;
            const uint32_t so = bx < by ? s : swap_state(s);
            if (st[p][q] && st[p][q] != so) ok = false;
            st[p][q] = so;
        }
        if (!ok) continue;
        unsigned long long maps;
        if (nb == 2) {
            maps = st[0][1] == 3u ? a.p5.small[14] : a.p5.small[13];
        } else {
            uint32_t code = 0;
            for (int p = 0; p < nb; p++)
                for (int q = p + 1; q < nb; q++) {
                    if (st[p][q] & 1u) code |= 1u << code_bit(nb, p, q);
                    if (st[p][q] & 2u) code |= 1u << code_bit(nb, q, p);
                }
            const int c = (int)(nb == 3 ? __ldg(a.p5.lut3_canon + code) : __ldg(a.p5.lut4_canon + code));
            if (c < 0) {
                set_status(a.status, ACC_ERR_INTERNAL);
                continue;
            }
            if (nb == 3) {
                maps = a.p5.small[c] * a.p5.aut3[c];
            } else {
                // (a triangle with a pendant is kept doubled, see partial.cu)
                int edges = 0, deg[4] = {};
                for (int p = 0; p < 4; p++)
                    for (int q = p + 1; q < 4; q++)
                        if (st[p][q]) {
                            edges++;
                            deg[p]++;
                            deg[q]++;
                        }
                const bool paw = edges == 4 && (deg[0] == 3 || deg[1] == 3 || deg[2] == 3 || deg[3] == 3);
                const unsigned long long P = a.part[c];
                maps = (paw ? P >> 1 : P) * a.p5.aut4[c];
            }
        }
        if (!maps) continue;
        const int to = (int)__ldg(a.p5.lut5 + code5);
        if (to < 0) set_status(a.status, ACC_ERR_INTERNAL);
        else atomicAdd(&a.p5.sums[to], 0ull - maps);
    }
}

// Inclusion and exclusion: class c with partial count P adds (-1)^(edges left
// out) P to the class of every subset of its edges that connects the five
// vertices.  Warp per class, a lane a subset: 12 to 30 us by the classes present.
__global__ void __launch_bounds__(256) k_counts5(PartialArgs a) {
    grid_dep_wait();
    __shared__ int instead;
    ask_scan(a, &instead);
    extern __shared__ __align__(16) unsigned char smem[];
    Bins5 bins = bins5(a, reinterpret_cast<uint32_t *>(smem));
    bins.sums = a.counts;
    bins.clear();
    if (instead) return;
    const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), warps = (int)((gridDim.x * blockDim.x) >> 5),
              lane = threadIdx.x & 31;
    for (int c = warp; c < kN5; c += warps) {
        const unsigned long long sum = a.p5.sums[c];
        if (!sum) continue;
        const unsigned long long P = sum / a.p5.div5[c];
        if (P * a.p5.div5[c] != sum) {
            set_status(a.status, ACC_ERR_INTERNAL);
            continue;
        }
        const uint32_t code = a.p5.code5[c];
        uint32_t edge[10];
        int n = 0;
        for (int i = 0; i < 5; i++)
            for (int j = i + 1; j < 5; j++) {
                const uint32_t bits = code & ((1u << code_bit(5, i, j)) | (1u << code_bit(5, j, i)));
                if (bits) edge[n++] = bits;
            }
        for (uint32_t sub = lane; sub < 1u << n; sub += kWarp) {
            uint32_t kept = 0;
            for (int e = 0; e < n; e++) kept |= (sub >> e) & 1u ? edge[e] : 0u;
            const int to = (int)__ldg(a.p5.lut5_canon + kept);
            if (to >= 0) bins.add_class(to, (n - __popc(sub)) & 1 ? 0ull - P : P);
        }
    }
    bins.flush();
}

bool launched() {
    if (cudaPeekAtLastError() == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

int share(int per_sm, int num_sms, int grid_num, int grid_den) {
    const long long g = (long long)num_sms * per_sm * grid_num / grid_den;
    return (int)(g < num_sms ? num_sms : g);
}

}  // namespace

void partial5_tables(const uint32_t *code5, const uint32_t *code4, const uint32_t *code3, std::vector<unsigned char> &div5,
                     std::vector<unsigned char> &aut4, std::vector<unsigned char> &aut3) {
    div5.assign(kN5, 1);
    for (int c = 0; c < kN5; c++) {
        bool adj[5][5] = {};
        int deg[5] = {}, n[5] = {}, edges = 0, tri = 0;
        for (int i = 0; i < 5; i++)
            for (int j = i + 1; j < 5; j++)
                if (code5[c] & ((1u << code_bit(5, i, j)) | (1u << code_bit(5, j, i)))) {
                    adj[i][j] = adj[j][i] = true;
                    deg[i]++;
                    deg[j]++;
                    edges++;
                }
        for (int i = 0; i < 5; i++) n[deg[i]]++;  // vertices by degree
        for (int i = 0; i < 5; i++)
            for (int j = i + 1; j < 5; j++)
                for (int k = j + 1; k < 5; k++) tri += adj[i][j] && adj[j][k] && adj[i][k];
        int d = 1;
        if (edges == 4) d = n[4] ? 1 : 2;                           // star; fork, path
        else if (edges == 5) d = n[2] == 5 ? 1 : (n[4] ? 4 : 2);    // cycle; triangle with two pendants at a vertex; others
        else if (edges == 6) d = n[4] == 1 && n[2] == 4 ? 8 : (n[3] == 2 && n[2] == 3 && !tri ? 1 : 2);  // two triangles; K_{2,3}
        else if (edges == 7) d = n[4] == 1 && n[3] == 2 && n[2] == 2 ? 2 : 1;  // fan; the others directly
        else if (edges == 8) d = n[4] == 1 ? 4 : 1;                 // wheel; K_4 with a vertex on two of its vertices
        else if (edges == 9) d = 3;
        div5[c] = (unsigned char)d;
    }
    auto automorphisms = [](int k, uint32_t code) -> int {
        int p[5] = {0, 1, 2, 3, 4}, count = 0;
        auto same = [&]() {
            for (int i = 0; i < k; i++)
                for (int j = 0; j < k; j++)
                    if (i != j && ((code >> code_bit(k, i, j)) & 1u) != ((code >> code_bit(k, p[i], p[j])) & 1u)) return false;
            return true;
        };
        const int total = k == 3 ? 6 : 24;
        for (int x = 0; x < total; x++) {  // the x-th permutation by insertion
            int y = x;
            for (int i = 0; i < k; i++) {
                const int at = i - y % (i + 1);
                y /= i + 1;
                for (int j = i; j > at; j--) p[j] = p[j - 1];
                p[at] = i;
            }
            count += same();
        }
        return count;
    };
    aut3.resize(num_classes(3));
    aut4.resize(num_classes(4));
    for (int c = 0; c < num_classes(3); c++) aut3[c] = (unsigned char)automorphisms(3, code3[c]);
    for (int c = 0; c < num_classes(4); c++) aut4[c] = (unsigned char)automorphisms(4, code4[c]);
}

int launch_partial5(PartialArgs &a, long long max_entries, int num_sms, cudaStream_t s, int grid_num, int grid_den) {
    static std::atomic<unsigned long long> limit[2];
    if (!raise_shared_limit(k_cycles5<1>, cycle_smem(1), limit[0]) || !raise_shared_limit(k_cycles5<2>, cycle_smem(2), limit[1]))
        return ACC_ERR_CUDA;
    // Most of these passes wait on memory or on their last few blocks, so they run
    // side by side where the data allows (JoinsPrevious): the 5-cycles beside the
    // wedges of k = 4, then the pairs' first phase beside the finish, then its second
    // beside the products (5000 vertices, regulatory: 506 us one
    // after another, 459 side by side; 1899 vertices, 20296 arcs: 1657 and 1411).
    int launches = launch_partial5_prep(a, max_entries, num_sms, s);
    if (launches < 0) return launches;
    const int grid = share(3, num_sms, grid_num, grid_den);
    launch_pdl(k_cycles5<1>, grid, kCThreads, cycle_smem(1), s, a);
    if (!launched()) return ACC_ERR_CUDA;
    int rc = launch_partial5_wedges(a, 1, num_sms, s, grid_num, grid_den);
    if (rc < 0) return rc;
    launch_pdl(k_cycles5<2>, share(2, num_sms, grid_num, grid_den), kCThreads, cycle_smem(2), s, a);
    if (!launched()) return ACC_ERR_CUDA;
    rc = launch_partial5_wedges(a, 2, num_sms, s, grid_num, grid_den);
    if (rc < 0) return rc;
    rc = launch_partial5_pairs(a, 1, num_sms, s, grid_num, grid_den);
    if (rc < 0) return rc;
    rc = launch_partial5_finish(a, max_entries, num_sms, s);
    if (rc < 0) return rc;
    rc = launch_partial5_pairs(a, 2, num_sms, s, grid_num, grid_den);
    if (rc < 0) return rc;
    launches += 7;
    int tiles = (a.gs.one.n + kVTile - 1) / kVTile;
    if (tiles > 2 * num_sms) tiles = 2 * num_sms;
    launch_pdl(k_vertex5, tiles < 1 ? 1 : tiles, kVThreads, 0, s, a);
    if (!launched()) return ACC_ERR_CUDA;
    launch_pdl(k_closed5, share(2, num_sms, grid_num, grid_den), 256, kN5 * 4, s, a);
    if (!launched()) return ACC_ERR_CUDA;
    if (a.nh) launch_pdl(k_diamonds5<true>, share(2, num_sms, grid_num, grid_den), 256, kN5 * 4, s, a);
    else launch_pdl(k_diamonds5<false>, share(2, num_sms, grid_num, grid_den), 256, kN5 * 4, s, a);
    if (!launched()) return ACC_ERR_CUDA;
    launch_pdl(k_quotients, num_sms * 4, 256, 0, s, a);
    return launched() ? launches + 4 : ACC_ERR_CUDA;
}

int launch_partial5_counts(const PartialArgs &a, int num_sms, cudaStream_t s) {
    launch_pdl(k_counts5, num_sms * 4, 256, kN5 * 4, s, a);
    return launched() ? 1 : ACC_ERR_CUDA;
}

}  // namespace acc
