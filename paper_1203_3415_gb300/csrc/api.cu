// C ABI: context, workspace and the counting entry points.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <mutex>
#include <new>
#include <vector>

#include "common.cuh"
#include "context.cuh"
#include "formula.cuh"
#include "partial.cuh"
#include "randomise.cuh"

using namespace acc;

namespace {

#ifndef ACC_QUEUE_CAP
#define ACC_QUEUE_CAP (1ull << 22)
#endif
constexpr unsigned long long kQueueCap = ACC_QUEUE_CAP;
// ACC_ADJ_AUTO: count-mode probes read hashed tables for sets whose largest
// graph has at least this many vertices (k = 5; k = 3, 4), where the dense
// block's probes (n^2/4 bytes, out of L2) get slower than the hashed ones
// (measured on GB300: k = 5 dense/hashed 82/87 scanned entries per ns at
// n = 40000, 53/87 at 80000; k = 4 149/107 at 40000, 122/108 at 80000).
constexpr int kHashMinN5 = 49152;
constexpr int kHashMinN34 = 131072;
bool hash_auto(int k, int max_n) { return max_n >= (k == 5 ? kHashMinN5 : kHashMinN34); }
// Below this many vertices the renumbering pass costs more than it saves.
constexpr int kRelabelMinN = 1024;
// ACC_MODE_AUTO: largest graph (vertices) for which k = 3 takes the formula path.
constexpr int kAutoFormulaMaxN = 16384;

bool ok(cudaError_t e) { return e == cudaSuccess; }

// Whether the last failed allocation met a stream capture, not a lack of memory.
thread_local bool t_alloc_in_capture = false;

template <typename T>
int grow(T **p, size_t *cap, size_t need) {
    if (need <= *cap && *p) return ACC_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    const size_t alloc = need + need / 4 + 64;
    const cudaError_t e = cudaMalloc((void **)p, alloc * sizeof(T));
    if (!ok(e)) {
        cudaGetLastError();
        *p = nullptr;
        t_alloc_in_capture = e == cudaErrorStreamCaptureUnsupported;
        return ACC_ERR_NOMEM;
    }
    *cap = alloc;
    return ACC_OK;
}

bool valid_k(int k) { return k >= 3 && k <= 5; }

// Class tables are built once per device and k and shared by every context
// on that device (the request server runs one context per slot); each
// context holds a reference, and the last one released frees the table.
struct SharedTable {
    int refs = 0;
    int16_t *lut = nullptr, *lut_sv = nullptr;
    uint32_t *class_code = nullptr;
    uint32_t *inv = nullptr;  // k = 3, 4: partial_matrix
    unsigned char *tab5 = nullptr;  // k = 5: partial5_tables
    int16_t *lut_host = nullptr;
    uint32_t *class_code_host = nullptr;
};
constexpr int kTableDevices = 64;
SharedTable g_tables[kTableDevices][6];
std::mutex g_tables_mu;

// Build the table for k on stream s (waits for it) into t; on failure t is
// left empty.
int build_table(int k, cudaStream_t s, SharedTable &t) {
    const size_t ncodes = size_t(1) << code_bits(k);
    const int ncls = num_classes(k);
    uint32_t *canon = nullptr;
    int *rank = nullptr;
    int16_t *lut = nullptr, *lut_sv = nullptr;
    uint32_t *cc = nullptr, *inv = nullptr;
    int16_t *lut_host = new (std::nothrow) int16_t[ncodes];
    uint32_t *cc_host = new (std::nothrow) uint32_t[ncls];
    int rc = ACC_ERR_NOMEM;
    if (!lut_host || !cc_host) goto fail;
    if (!ok(cudaMalloc(&canon, ncodes * 4)) || !ok(cudaMalloc(&rank, (size_t)rank_ints(k) * 4)) ||
        !ok(cudaMalloc(&lut, ncodes * 2)) || !ok(cudaMalloc(&lut_sv, ncodes * 2)) ||
        !ok(cudaMalloc(&cc, ncls * 4)))
        goto fail;
    rc = launch_build_lut(k, canon, rank, lut, cc, lut_sv, s);
    if (rc < 0) goto fail;
    rc = ACC_ERR_CUDA;
    if (!ok(cudaMemcpyAsync(lut_host, lut, ncodes * 2, cudaMemcpyDeviceToHost, s))) goto fail;
    if (!ok(cudaMemcpyAsync(cc_host, cc, ncls * 4, cudaMemcpyDeviceToHost, s))) goto fail;
    if (!ok(cudaStreamSynchronize(s))) goto fail;
    {
        // the table must use every class index exactly up to ncls - 1
        int mx = -1;
        for (size_t i = 0; i < ncodes; i++) {
            if (lut_host[i] < -1) mx = 1 << 20;
            if (lut_host[i] > mx) mx = lut_host[i];
        }
        if (mx != ncls - 1) {
            rc = ACC_ERR_INTERNAL;
            goto fail;
        }
    }
    if (k <= 4) {
        std::vector<uint32_t> m;
        partial_matrix(k, lut_host, cc_host, m);
        if (!ok(cudaMalloc(&inv, m.size() * 4)) ||
            !ok(cudaMemcpyAsync(inv, m.data(), m.size() * 4, cudaMemcpyHostToDevice, s)) ||
            !ok(cudaStreamSynchronize(s))) {
            rc = inv ? ACC_ERR_CUDA : ACC_ERR_NOMEM;
            goto fail;
        }
    }
    cudaFree(canon);
    cudaFree(rank);
    t.lut = lut;
    t.lut_sv = lut_sv;
    t.class_code = cc;
    t.inv = inv;
    t.lut_host = lut_host;
    t.class_code_host = cc_host;
    return ACC_OK;
fail:
    cudaGetLastError();
    cudaFree(canon);
    cudaFree(rank);
    cudaFree(lut);
    cudaFree(lut_sv);
    cudaFree(cc);
    cudaFree(inv);
    delete[] lut_host;
    delete[] cc_host;
    return rc;
}

int ensure_lut(acc_ctx *c, int k, cudaStream_t s);

// k = 5 by partial patterns reads the tables of every k, and each class's
// divisor and the smaller classes' automorphisms (built with the k = 5 table).
int ensure_tab5(acc_ctx *c, cudaStream_t s) {
    for (int k = 5; k >= 3; k--) {
        const int rc = ensure_lut(c, k, s);
        if (rc) return rc;
    }
    if (c->tab5) return ACC_OK;
    std::lock_guard<std::mutex> lock(g_tables_mu);
    SharedTable &t = g_tables[c->device][5];
    if (!t.tab5) {
        std::vector<unsigned char> div5, aut4, aut3;
        partial5_tables(c->class_code_host[5], c->class_code_host[4], c->class_code_host[3], div5, aut4, aut3);
        div5.insert(div5.end(), aut4.begin(), aut4.end());
        div5.insert(div5.end(), aut3.begin(), aut3.end());
        unsigned char *d = nullptr;
        if (!ok(cudaMalloc(&d, div5.size()))) {
            cudaGetLastError();
            return ACC_ERR_NOMEM;
        }
        if (!ok(cudaMemcpyAsync(d, div5.data(), div5.size(), cudaMemcpyHostToDevice, s)) || !ok(cudaStreamSynchronize(s))) {
            cudaGetLastError();
            cudaFree(d);
            return ACC_ERR_CUDA;
        }
        t.tab5 = d;
    }
    c->tab5 = t.tab5;  // (the context holds a reference to the k = 5 table)
    return ACC_OK;
}

int ensure_lut(acc_ctx *c, int k, cudaStream_t s) {
    if (c->lut[k]) return ACC_OK;
    if (c->device < 0 || c->device >= kTableDevices) return ACC_ERR_ARG;
    std::lock_guard<std::mutex> lock(g_tables_mu);
    SharedTable &t = g_tables[c->device][k];
    if (t.refs == 0) {
        const int rc = build_table(k, s, t);
        if (rc) return rc;
    }
    t.refs++;
    c->lut[k] = t.lut;
    c->lut_sv[k] = t.lut_sv;
    c->class_code_dev[k] = t.class_code;
    c->inv[k] = t.inv;
    c->lut_host[k] = t.lut_host;
    c->class_code_host[k] = t.class_code_host;
    return ACC_OK;
}

// Drop the context's references to the shared tables (the device is current).
void release_luts(acc_ctx *c) {
    std::lock_guard<std::mutex> lock(g_tables_mu);
    for (int k = 3; k <= 5; k++) {
        if (!c->lut[k]) continue;
        SharedTable &t = g_tables[c->device][k];
        if (--t.refs == 0) {
            cudaFree(t.lut);
            cudaFree(t.lut_sv);
            cudaFree(t.class_code);
            cudaFree(t.inv);
            cudaFree(t.tab5);
            delete[] t.lut_host;
            delete[] t.class_code_host;
            t = SharedTable();
        }
        c->lut[k] = c->lut_sv[k] = nullptr;
        c->class_code_dev[k] = nullptr;
        c->inv[k] = nullptr;
        if (k == 5) c->tab5 = nullptr;
        c->lut_host[k] = nullptr;
        c->class_code_host[k] = nullptr;
    }
}

// per warp: two overflow lists of up to max_n entries, then the k = 5 count
// mode's collected part-B rows
long long scratch_per_warp(int max_n) { return 2 * (((long long)max_n + 32 + 31) & ~31LL) + 2 * kPartBRows; }

// The count mode, and the automatic mode that runs it for k = 4, 5 and for
// any graph above the dense block's limit.
bool count_family(const acc_ctx *c) { return c->mode == ACC_MODE_COUNT || c->mode == ACC_MODE_AUTO; }

// The count mode builds the lists without the dense block (and probes
// hashed tables) above the dense block's limit, or when asked to.
bool sparse_build(const acc_ctx *c, int max_n) {
    return count_family(c) && (c->adjacency == ACC_ADJ_SPARSE || max_n > ACC_MAX_N);
}

bool uses_hash(const acc_ctx *c, int k, int max_n) {
    return count_family(c) &&
           (c->adjacency == ACC_ADJ_HASH || c->adjacency == ACC_ADJ_SPARSE || max_n > ACC_MAX_N ||
            (c->adjacency == ACC_ADJ_AUTO && hash_auto(k, max_n)));
}

// The count mode's scans stage the list rows that are neighbours of the
// root from the reverse positions of the root's entries (ACC_REV=0 at build
// time: by binary search, as for every other row).  Sets of fewer than
// ACC_REV_MIN_ARCS arcs skip them: building them costs about 4 us, more than
// the searches they save on small graphs (k = 3 count on 1000 vertices and
// 5000 arcs: 0.035 ms per count without, 0.039 with; k = 4 on 20000 vertices
// and 100000 arcs: 0.604 without, 0.572 with).
#ifndef ACC_REV
#define ACC_REV 1
#endif
#ifndef ACC_REV_MIN_ARCS
#define ACC_REV_MIN_ARCS 8192
#endif
bool uses_rev(const acc_ctx *c, long long arcs) { return ACC_REV && count_family(c) && arcs >= ACC_REV_MIN_ARCS; }

// The automatic mode takes the k = 3 formula path on graphs of up to
// kAutoFormulaMaxN vertices (measured faster there than the count mode's
// scan: 0.028 against 0.034 ms at 1000 vertices, 0.065 against 0.100 at 5000;
// slower at 20000 with hubs of degree 470, 0.208 against 0.181).
bool uses_formula(const acc_ctx *c, int k, int max_n) {
    return c->mode == ACC_MODE_FORMULA || (c->mode == ACC_MODE_AUTO && k == 3 && max_n <= kAutoFormulaMaxN &&
                                           !sparse_build(c, max_n) && !uses_hash(c, k, max_n));
}

// The count mode of k = 3, 4 counts by partial patterns (partial.cu) on sets
// whose vertices are renumbered by degree, from ACC_PARTIAL_MIN_ARCS arcs on
// for k = 3 and sets of several graphs, from ACC_PARTIAL_MIN_ARCS1 for one graph
// of k = 4: the passes of a small graph take longer than its list scan
// (scan / partial, us: k = 4, 8300 arcs on 4000 vertices 60 / 69 uniform, 73 / 82
// with hubs; 12000 on 3000 65 / 67 and 117 / 104; 20000 on 5000 78 / 80 and 199 /
// 119).  Only n and m are known here.  From 12288 to about 32000 arcs, graphs of 1 to
// 3 arcs a vertex with light tails still lose (12600 on 12000 vertices, uniform 74 /
// 83, degrees up to 25 76 / 92; 24000 on 12000, up to 25, 91 / 99), and those with hubs
// gain more (up to 60 115 / 102; up to 100, 12400 on 6000, 126 / 98; up to 1000, 30000
// on 20000, 260 / 148).
#ifndef ACC_PARTIAL_MIN_ARCS
#define ACC_PARTIAL_MIN_ARCS 8192
#endif
#ifndef ACC_PARTIAL_MIN_ARCS1
#define ACC_PARTIAL_MIN_ARCS1 (ACC_PARTIAL_MIN_ARCS * 3 / 2)
#endif
// Many tiny graphs: the finish takes a block a graph, and its fixed part (the
// graph's sums, its class matrix) more than the scan of the graph does.  Sets of
// more graphs than the finish has blocks at once are scanned below 64 arcs a graph
// (96 where the graphs have fewer than 32 vertices; scan / partial, us, k = 4: 4000
// graphs of 10 vertices and 20 arcs 267 / 368, of 40 and 40 326 / 400, of 20 and
// 80 487 / 524, of 40 and 80 468 / 450, of 80 and 160 747 / 567; 300 graphs of 20
// and 40 97 / 82).  k = 3, whose finish is short: from 16 graphs an SM on, below 48
// (16000 graphs of 20 vertices and 40 arcs 792 / 837, of 40 and 80 1001 / 968).
bool tiny_graphs(const acc_ctx *c, int k, int max_n, long long arcs, int B) {
    return k == 3 ? B > 16 * c->num_sms && arcs < 48ll * B
                  : B > 4 * c->num_sms && arcs < (max_n < 32 ? 96ll : 64ll) * B;
}

bool uses_partial(const acc_ctx *c, int k, int max_n, long long arcs, bool relabel, int B) {
    return count_family(c) && k <= 4 && relabel && arcs < c->partial_arcs_end && !uses_formula(c, k, max_n) &&
           arcs >= (k == 4 && B == 1 ? ACC_PARTIAL_MIN_ARCS1 : ACC_PARTIAL_MIN_ARCS) &&
           !tiny_graphs(c, k, max_n, arcs, B);
}

// The same for k = 5 (partial5.cu), of one graph; its launches are followed by
// the scan's, which run only when the device finds that it must (more
// triangles than the list holds, a root with over kCycleRows neighbours above it,
// left_to_scan).
// From ACC_PARTIAL_MIN_ARCS arcs on, of at least two a vertex below
// ACC_PARTIAL_MIN_ARCS1 (scan / partial, us: 8300 uniform arcs on 4000 vertices 182 /
// 150, 9000 on 6000 105 / 145).  Only n and m are known here: graphs with hubs below
// the line would gain too (820 / 312 and 702 / 246 at those sizes).
bool uses_partial5(const acc_ctx *c, int k, int n, long long arcs, bool relabel, int B) {
    return count_family(c) && k == 5 && B == 1 && relabel && arcs < c->partial_arcs_end && arcs >= ACC_PARTIAL_MIN_ARCS &&
           (arcs >= 2ll * n || arcs >= ACC_PARTIAL_MIN_ARCS1);
}

// One graph counted by partial patterns that is large enough for its dense block
// to cost more than sorted rows and hashed tables do takes the sparse build
// (ACC_ADJ_AUTO).  Measured, dense / sparse, us: k = 3, 250000 arcs on 50000
// vertices 221 / 235 with hubs, 164 / 152 uniform; 300000 on 100000 296 / 212 and
// 218 / 155; k = 4, 260000 on 66000 361 / 381 and 229 / 202; 200000 on 100000 298 /
// 248 and 205 / 162.  Up to kSparseArcs arcs a vertex, above which the rows' sort and
// the hashed probes take longer than the block (98304 vertices, with hubs of up to
// 500, 1000 and 2000, and uniform: 10 a vertex k = 3 604 / 489 and 499 / 306, k = 4
// 1610 / 1670 and 860 / 702; 20 a vertex k = 3 1070 / 1097 and 848 / 667, k = 4 6647 /
// 8955 and 2179 / 2036; 40 a vertex k = 3 2231 / 3007 and 1681 / 1468; 100 a vertex,
// uniform, k = 3 4637 / 6290).
constexpr long long kSparseArcs[5] = {0, 0, 0, 20, 10};
#ifndef ACC_SPARSE_MIN_N
#define ACC_SPARSE_MIN_N 98304
#endif
bool sparse_auto(const acc_ctx *c, int k, int max_n, long long arcs, bool relabel, int B) {
    return c->adjacency == ACC_ADJ_AUTO && B == 1 && max_n >= ACC_SPARSE_MIN_N && k <= 4 &&
           (c->sparse_any || arcs <= kSparseArcs[k] * max_n) &&
           uses_partial(c, k, max_n, arcs, relabel, B);
}
bool sparse_path(const acc_ctx *c, int k, int max_n, long long arcs, bool relabel, int B) {
    return sparse_build(c, max_n) || sparse_auto(c, k, max_n, arcs, relabel, B);
}
// The sparse build waits for the largest degree, which sizes the scan's
// overflow lists; partial patterns have none, and hold any degree of a graph of
// kNdMax vertices.
bool sparse_waits(const acc_ctx *c, int k, int max_n, long long arcs, bool relabel, int B) {
    return !(uses_partial(c, k, max_n, arcs, relabel, B) && max_n <= kNdMax);
}

// Size limit of one graph: the dense block's, or the sparse build's for the
// count mode (local ids fill 26 bits of the extension-list entries).
int size_check(const acc_ctx *c, long long n) {
    if (n > ACC_MAX_N_SPARSE) return ACC_ERR_TOO_LARGE;
    if (n > ACC_MAX_N && !count_family(c)) return ACC_ERR_TOO_LARGE;
    return ACC_OK;
}

// Entries of one per-warp overflow list for the sparse build: an extension
// list holds at most 3 maxdeg vertices (k = 5: the level-2 list after w2
// and the neighbours of w2; k = 4: two neighbour lists; k = 3: one).
long long sparse_list_entries(int maxdeg) { return (3LL * maxdeg + 64 + 31) & ~31LL; }

// What a set of NV vertices in a dense block of `words` words, with at most `arcs`
// arcs and graphs of at most max_n vertices, needs: need(&buffer, &capacity,
// elements) for each buffer.  (The sparse build's overflow lists are sized by the
// largest degree, once it is known: run_set.)  either: for the list scan and, where a
// set of no more arcs may take them, the partial patterns.
template <typename Need>
void workspace_needs(acc_ctx *c, long long NV, long long words, long long arcs, int max_n, int k, int B, bool relabel,
                     int warps, bool either, Need need) {
    const bool sparse = sparse_path(c, k, max_n, arcs, relabel, B);
    const bool may = either && count_family(c) && relabel && arcs >= ACC_PARTIAL_MIN_ARCS && arcs < c->partial_arcs_end;
    const bool partial = uses_partial(c, k, max_n, arcs, relabel, B) || (may && k <= 4);
    const bool partial5 = uses_partial5(c, k, max_n, arcs, relabel, B) || (may && k == 5 && B == 1);
    const size_t n1 = (size_t)NV + 1, entries = (size_t)(2 * arcs);
    if (partial5) {
        need(&c->p5_vert, &c->p5_vert_cap, 3 * n1);
        need(&c->p5_sums, &c->p5_sums_cap, (size_t)num_classes(5) + 16 + kCtrs);
    }
    if (partial || partial5) {
        need(&c->pp_nd, &c->pp_nd_cap, n1);
        need(&c->pp_part, &c->pp_part_cap, (size_t)B * num_classes(k == 5 ? 4 : k));
        need(&c->pp_done, &c->pp_done_cap, (size_t)B);
        if (k >= 4) need(&c->pp_wedges, &c->pp_wedges_cap, n1);
        if (k >= 4) need(&c->pp_tri, &c->pp_tri_cap, 3 * entries + 1);
    }
    if (sparse || uses_hash(c, k, max_n)) need(&c->nh, &c->nh_cap, (size_t)kNhWords * entries + 4);
    if (sparse) {
        need(&c->sp_raw, &c->sp_raw_cap, entries + 1);
        need(&c->sp_merged, &c->sp_merged_cap, entries + 1);
        need(&c->sp_roff, &c->sp_roff_cap, n1);
        need(&c->sp_big, &c->sp_big_cap, (size_t)sparse_big_rows_cap(arcs));
    } else {
        need(&c->state, &c->state_cap, (size_t)words + 4);
        need(&c->occ, &c->occ_cap, (size_t)NV * (size_t)occ_words(max_n) + 1);
    }
    need(&c->deg, &c->deg_cap, n1);
    need(&c->lo, &c->lo_cap, n1);
    need(&c->nptr, &c->nptr_cap, n1);
    need(&c->label, &c->label_cap, n1);
    need(&c->deg_in, &c->deg_in_cap, n1);
    need(&c->tiles, &c->tiles_cap, (size_t)scan_tiles_needed(NV) + 1);
    need(&c->f5_pre, &c->f5_pre_cap, n1);
    need(&c->nbr, &c->nbr_cap, entries + 1);
    need(&c->src, &c->src_cap, entries + 1);
    if (uses_rev(c, arcs) || (partial && k == 4) || partial5) need(&c->rev, &c->rev_cap, entries + 1);
    // (partial patterns have no extension lists)
    if (!sparse && (!partial || either)) need(&c->scratch, &c->scratch_cap, (size_t)scratch_per_warp(max_n) * (size_t)warps);
}

// Every buffer that workspace_needs may ask for: each(&buffer, &capacity).
template <typename Each>
void workspace_buffers(acc_ctx *c, Each each) {
    each(&c->p5_vert, &c->p5_vert_cap);
    each(&c->p5_sums, &c->p5_sums_cap);
    each(&c->pp_nd, &c->pp_nd_cap);
    each(&c->pp_part, &c->pp_part_cap);
    each(&c->pp_done, &c->pp_done_cap);
    each(&c->pp_wedges, &c->pp_wedges_cap);
    each(&c->pp_tri, &c->pp_tri_cap);
    each(&c->nh, &c->nh_cap);
    each(&c->sp_raw, &c->sp_raw_cap);
    each(&c->sp_merged, &c->sp_merged_cap);
    each(&c->sp_roff, &c->sp_roff_cap);
    each(&c->sp_big, &c->sp_big_cap);
    each(&c->state, &c->state_cap);
    each(&c->occ, &c->occ_cap);
    each(&c->deg, &c->deg_cap);
    each(&c->lo, &c->lo_cap);
    each(&c->nptr, &c->nptr_cap);
    each(&c->label, &c->label_cap);
    each(&c->deg_in, &c->deg_in_cap);
    each(&c->tiles, &c->tiles_cap);
    each(&c->f5_pre, &c->f5_pre_cap);
    each(&c->nbr, &c->nbr_cap);
    each(&c->src, &c->src_cap);
    each(&c->rev, &c->rev_cap);
    each(&c->scratch, &c->scratch_cap);
}

int grow_workspace(acc_ctx *c, long long NV, long long words, long long arcs, int max_n, int k, int B, bool relabel,
                   cudaStream_t s, bool either) {
    const int warps = enum_grid_warps(k, c->num_sms);
    if (warps < 0) return warps;
    int rc = ACC_OK;
    // a reallocation (the capacity changes; the address may not) brings
    // memory that is not zero: the next build sweeps it
    const size_t state_before = c->state_cap;
    workspace_needs(c, NV, words, arcs, max_n, k, B, relabel, warps, either, [&](auto **p, size_t *cap, size_t need) {
        if (!rc) rc = grow(p, cap, need);
    });
    if (c->state_cap != state_before) c->state_clean = false;
    if (rc) return rc;
    if (!c->info) {
        if (!ok(cudaMalloc(&c->info, sizeof(GraphInfo)))) return ACC_ERR_NOMEM;
        if (!ok(cudaMemsetAsync(c->info, 0, sizeof(GraphInfo), s))) return ACC_ERR_CUDA;
    }
    if (!c->queue) {
        if (!ok(cudaMalloc(&c->queue, kQueueCap * sizeof(uint4)))) return ACC_ERR_NOMEM;
        c->queue_cap = kQueueCap;
    }
    if (!c->status_dev) {
        if (!ok(cudaMalloc(&c->status_dev, sizeof(int)))) return ACC_ERR_NOMEM;
    }
    if (!c->maxdeg_host && !ok(cudaMallocHost(&c->maxdeg_host, sizeof(int)))) return ACC_ERR_NOMEM;
    return ACC_OK;
}

template <typename T>
void drop(T **p, size_t *cap) {  // (a free waits for the device)
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
}

// The launch graph may hold the addresses of buffers that are given back.
void drop_launch_graph(acc_ctx *c) {
    if (c->cg_exec) cudaGraphExecDestroy(c->cg_exec);
    c->cg_exec = nullptr;
    memset(&c->cg_seen, 0, sizeof(c->cg_seen));
}

// Gives back what only partial patterns need, with the sparse build's buffers.
void free_partial(acc_ctx *c, bool sparse) {
    drop_launch_graph(c);
    drop(&c->pp_nd, &c->pp_nd_cap);
    drop(&c->pp_part, &c->pp_part_cap);
    drop(&c->pp_done, &c->pp_done_cap);
    drop(&c->pp_wedges, &c->pp_wedges_cap);
    drop(&c->pp_tri, &c->pp_tri_cap);
    drop(&c->p5_vert, &c->p5_vert_cap);
    drop(&c->p5_sums, &c->p5_sums_cap);
    if (!sparse) return;
    drop(&c->nh, &c->nh_cap);
    drop(&c->sp_raw, &c->sp_raw_cap);
    drop(&c->sp_merged, &c->sp_merged_cap);
    drop(&c->sp_roff, &c->sp_roff_cap);
    drop(&c->sp_big, &c->sp_big_cap);
}

// The workspace of a set whose dense block has `words` words (see
// grow_workspace).  Where the device has no room for the way that the rules choose,
// another one is taken, for the context's later sets too (until the next
// acc_motif_prepare or acc_motif_batch_prepare): the sparse build for a graph
// that sparse_auto leaves to the dense block for its density, then the list scan for
// sets of as many arcs (partial patterns take 24 bytes a neighbour entry more, and
// the sparse build 40 more).
int ensure_workspace(acc_ctx *c, long long NV, long long words, long long arcs, int max_n, int k, int B, bool relabel,
                     cudaStream_t s, bool either = false) {
    int rc = grow_workspace(c, NV, words, arcs, max_n, k, B, relabel, s, either);
    if (rc != ACC_ERR_NOMEM || t_alloc_in_capture) return rc;
    bool sparse = sparse_path(c, k, max_n, arcs, relabel, B);
    if (!sparse && !c->sparse_any) {
        c->sparse_any = true;
        if (sparse_path(c, k, max_n, arcs, relabel, B)) {
            drop_launch_graph(c);
            drop(&c->state, &c->state_cap);
            drop(&c->occ, &c->occ_cap);
            c->state_clean = false;
            rc = grow_workspace(c, NV, words, arcs, max_n, k, B, relabel, s, either);
            if (rc != ACC_ERR_NOMEM) return rc;
            sparse = true;
        } else {
            c->sparse_any = false;
        }
    }
    if (!(either || uses_partial(c, k, max_n, arcs, relabel, B) || uses_partial5(c, k, max_n, arcs, relabel, B))) return rc;
    c->partial_arcs_end = arcs;
    free_partial(c, sparse && !sparse_path(c, k, max_n, arcs, relabel, B));
    return grow_workspace(c, NV, words, arcs, max_n, k, B, relabel, s, either);
}

// Build + enumerate one graph set into counts[B * num_classes(k)].
int run_set(acc_ctx *c, const GSet &gs, int max_n, int k, bool relabel, cudaStream_t s,
            int64_t *counts, int *status) {
    int launches = 0;
    c->timed_call = c->timing;
    if (c->timing && !ok(cudaEventRecord(c->ev[0], s))) return ACC_ERR_CUDA;
    const bool clean = c->state_clean;
    const bool sparse = sparse_path(c, k, max_n, gs.M, relabel, gs.B);
    if (!sparse) c->state_clean = false;  // until the closing clear below is enqueued
    // a buffer not known to be clean is swept whole (capacity, not just this
    // set's blocks): a later, larger set may use any part of it
    BuildBufs bb;
    bb.state = c->state;
    bb.state_words = (long long)c->state_cap;
    bb.state_clean = clean;
    bb.deg = c->deg;
    bb.lo = c->lo;
    bb.label = c->label;
    bb.deg_in = c->deg_in;
    bb.nptr = c->nptr;
    bb.tiles = c->tiles;
    bb.nbr = c->nbr;
    bb.src = c->src;
    bb.occ = c->occ;
    bb.occ_w = occ_words(max_n);
    bb.info = c->info;
    bb.k = k;
    bool partial = gs.NV > 0 && uses_partial(c, k, max_n, gs.M, relabel, gs.B);
    bool partial5 = gs.NV > 0 && uses_partial5(c, k, max_n, gs.M, relabel, gs.B);
    if (partial5) {
        if (!c->tab5) return ACC_ERR_INTERNAL;  // (the callers ensure it)
        bb.zero[4] = c->p5_vert;
        bb.nzero[4] = 3 * gs.NV;
        bb.zero[5] = reinterpret_cast<int *>(c->p5_sums);
        bb.nzero[5] = 2ll * (num_classes(5) + 16 + kCtrs);
    }
    if (partial || partial5) {
        bb.zero[0] = reinterpret_cast<int *>(c->pp_nd);
        bb.nzero[0] = 2 * gs.NV;
        bb.zero[1] = reinterpret_cast<int *>(c->pp_part);
        bb.nzero[1] = 2ll * gs.B * num_classes(k == 5 ? 4 : k);
        bb.zero[2] = c->pp_done;
        bb.nzero[2] = gs.B;
        if (k >= 4) {
            bb.zero[3] = reinterpret_cast<int *>(c->pp_wedges);
            bb.nzero[3] = gs.NV;
        }
    }
    int rc;
    if (sparse) {
        const SparseBufs sb = {c->sp_raw, c->sp_merged, c->sp_roff, c->sp_big};
        rc = launch_build_graph_sparse(gs, bb, sb, max_n, status, reinterpret_cast<unsigned long long *>(counts),
                                       (long long)gs.B * num_classes(k), relabel, c->num_sms, s);
    } else {
        rc = launch_build_graph(gs, bb, max_n, status, reinterpret_cast<unsigned long long *>(counts),
                                (long long)gs.B * num_classes(k), relabel, c->num_sms, s);
    }
    if (rc < 0) return rc;
    launches += rc;
    long long spw = scratch_per_warp(max_n);
    if (sparse && sparse_waits(c, k, max_n, gs.M, relabel, gs.B)) {
        // overflow lists sized by the largest degree: wait for the build
        if (!ok(cudaMemcpyAsync(c->maxdeg_host, &c->info->maxdeg, sizeof(int), cudaMemcpyDeviceToHost, s)) ||
            !ok(cudaStreamSynchronize(s)))
            return ACC_ERR_CUDA;
        if (*c->maxdeg_host > kNdMax) partial = partial5 = false;  // its packed degree counts hold kNdMax
        spw = 2 * sparse_list_entries(*c->maxdeg_host) + 2 * kPartBRows;
        const int warps = enum_grid_warps(k, c->num_sms);
        if (warps < 0) return warps;
        if (!partial && (rc = grow(&c->scratch, &c->scratch_cap, (size_t)spw * (size_t)warps))) return rc;
    }
    // count mode on a large set: probes read hashed tables, built from the
    // sorted neighbour lists
    const bool hash = gs.NV > 0 && (sparse || uses_hash(c, k, max_n));
    if (hash) {
        rc = launch_nh_build(c->nptr, c->deg, c->nbr, c->src, c->info, 2 * gs.M, c->nh, c->num_sms, s);
        if (rc < 0) return rc;
        launches += rc;
    }
    const bool formula = uses_formula(c, k, max_n);
    const bool rev = gs.NV > 0 && !formula && !partial && !partial5 && uses_rev(c, gs.M);
    if (rev) {
        rc = launch_rev_build(gs, c->nptr, c->deg, c->nbr, c->src, c->info, 2 * gs.M, c->rev, c->num_sms, s);
        if (rc < 0) return rc;
        launches += rc;
    }
    if (c->timing && !ok(cudaEventRecord(c->ev[1], s))) return ACC_ERR_CUDA;
    EnumArgs a;
    a.state = c->state;
    a.deg = c->deg;
    a.lo = c->lo;
    a.nptr = c->nptr;
    a.nbr = c->nbr;
    a.src = c->src;
    a.nh = hash ? reinterpret_cast<const uint4 *>(c->nh) : nullptr;
    a.rev = rev || partial5 ? c->rev : nullptr;
    a.lut = c->lut_sv[k];
    a.gs = gs;
    a.max_n = max_n;
    a.info = c->info;
    a.queue = c->queue;
    a.queue_cap = c->queue_cap;
    a.scratch = c->scratch;
    a.scratch_per_warp = spw;
    a.mode = c->mode == ACC_MODE_ENUMERATE ? 1 : 0;
    a.light = c->sched_light > 0 ? c->sched_light : enum_default_light(k, a.mode == 0);
    a.target = c->sched_target > 0 ? c->sched_target : enum_default_target(k, a.mode == 0);
    a.counts = reinterpret_cast<unsigned long long *>(counts);
    a.status = status;
    const bool any = gs.NV > 0;
    PartialArgs p = {};
    if (partial || partial5) {
        p.state = c->state;
        p.state_w = c->state;
        p.deg = c->deg;
        p.lo = c->lo;
        p.nptr = c->nptr;
        p.nbr = c->nbr;
        p.src = c->src;
        p.nh = hash ? c->nh : nullptr;
        p.lut = c->lut_sv[k == 5 ? 4 : k];
        p.inv = c->inv[k == 5 ? 4 : k];
        p.gs = gs;
        p.info = c->info;
        p.queue = c->queue;
        p.queue_cap = c->queue_cap;
        p.rev = c->rev;
        p.nd = c->pp_nd;
        p.wedges = c->pp_wedges;
        p.tri = c->pp_tri;
        p.part = c->pp_part;
        p.done = c->pp_done;
        p.counts = reinterpret_cast<unsigned long long *>(counts);
        p.status = status;
        p.occ = sparse ? nullptr : c->occ;
        p.occ_w = occ_words(max_n);
        if (partial5) {
            Partial5 &q = p.p5;
            q.sums = c->p5_sums;
            q.small = c->p5_sums + num_classes(5);
            q.ctr = q.small + 16;
            // the triangles are listed where the scan, if it runs after all,
            // keeps its overflow lists
            q.tris = reinterpret_cast<uint4 *>(c->scratch);
            q.tri_cap = c->scratch_cap / 4;
            q.in_tri = c->p5_vert;
            q.pair_wedges = reinterpret_cast<uint32_t *>(c->p5_vert + gs.NV);
            q.cycle_wedges = reinterpret_cast<uint32_t *>(c->p5_vert + 2 * gs.NV);
            q.lut5 = c->lut_sv[5];
            q.lut5_canon = c->lut[5];
            q.lut4_canon = c->lut[4];
            q.lut3 = c->lut_sv[3];
            q.lut3_canon = c->lut[3];
            q.code5 = c->class_code_dev[5];
            q.div5 = c->tab5;
            q.aut4 = c->tab5 + num_classes(5);
            q.aut3 = q.aut4 + num_classes(4);
            rc = launch_partial5(p, 2 * gs.M, c->num_sms, s, c->grid_num, c->grid_den);
        } else {
            rc = launch_partial(k, p, 2 * gs.M, c->num_sms, s, c->grid_num, c->grid_den);
        }
        if (rc < 0) return rc;
        launches += rc;
    }
    if (partial) {
        // counted
    } else if (any && formula) {
        if (k == 3)
            rc = launch_formula3(gs, c->state, c->nptr, c->deg, c->lo, c->nbr, c->lut[3],
                                 reinterpret_cast<unsigned long long *>(counts), status, c->num_sms, s);
        else if (k == 4)
            rc = launch_formula4(gs, c->state, c->nptr, c->deg, c->lo, c->nbr, c->lut[4], c->class_code_dev[4],
                                 c->info, reinterpret_cast<unsigned long long *>(counts), status, c->num_sms, s);
        else
            rc = launch_formula5(gs, c->state, c->nptr, c->deg, c->nbr, c->lut[5], c->class_code_dev[5], c->f5_pre,
                                 reinterpret_cast<unsigned long long *>(counts), status, c->num_sms, s);
        if (rc < 0) return rc;
        launches += rc;
    } else if (any) {
        rc = launch_enumerate(k, a, c->num_sms, 1, s, c->grid_num, c->grid_den);
        if (rc < 0) return rc;
        launches += rc;
    }
    if (c->timing && !ok(cudaEventRecord(c->ev[3], s))) return ACC_ERR_CUDA;
    if (any && !formula && !partial) {
        rc = launch_enumerate(k, a, c->num_sms, 2, s, c->grid_num, c->grid_den);
        if (rc < 0) return rc;
        launches += rc;
    }
    if (partial5) {
        rc = launch_partial5_counts(p, c->num_sms, s);
        if (rc < 0) return rc;
        launches += rc;
    }
    if (c->timing && !ok(cudaEventRecord(c->ev[2], s))) return ACC_ERR_CUDA;
    if (!sparse) {
        if (!partial) {  // (its last kernel clears the block)
            rc = launch_clear_graph(gs, c->state, c->occ, occ_words(max_n), c->num_sms, s);
            if (rc < 0) return rc;
            launches += rc;
        }
        c->state_clean = true;
    }
    c->last_launches = launches;
    c->last_partial5 = partial5;
    c->last_k = k;
    c->last_units = gs.NV;
    c->last_blocks = enum_grid_warps(k, c->num_sms) / kWarpsPerBlock * c->grid_num / c->grid_den;
    return ACC_OK;
}

// Wait for the call's device status when the caller gave no status word.
int finish(acc_ctx *c, cudaStream_t s, int32_t *status_user) {
    if (status_user) return ACC_OK;
    if (!ok(cudaMemcpyAsync(c->status_host, c->status_dev, sizeof(int), cudaMemcpyDeviceToHost, s)))
        return ACC_ERR_CUDA;
    if (!ok(cudaStreamSynchronize(s))) return ACC_ERR_CUDA;
    return *c->status_host;
}

int count_impl(acc_ctx *c, const int64_t *rowptr, const int32_t *col, int32_t n, int64_t m, int k,
               cudaStream_t s, int64_t *counts, int32_t *status_user) {
    if (!c || !rowptr || !counts || (m > 0 && !col)) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (n < 0 || m < 0 || m >= (1ll << 31)) return ACC_ERR_INPUT;
    if (size_check(c, n)) return ACC_ERR_TOO_LARGE;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    int rc = uses_partial5(c, k, n, m, n >= kRelabelMinN, 1) ? ensure_tab5(c, s) : ensure_lut(c, k, s);
    if (rc) return rc;
    const long long pitch = state_pitch(n);
    if ((rc = ensure_workspace(c, n, (long long)n * pitch, m, n, k, 1, n >= kRelabelMinN, s))) return rc;
    const bool sparse = sparse_path(c, k, n, m, n >= kRelabelMinN, 1);
    GSet gs = {};
    gs.one.rowptr = reinterpret_cast<const long long *>(rowptr);
    gs.one.col = col;
    gs.one.m = m;
    gs.one.soff = 0;
    gs.one.moff = 0;
    gs.one.pitch = pitch;
    gs.one.n = n;
    gs.one.voff = 0;
    gs.B = 1;
    gs.NV = n;
    gs.M = m;
    int *status = status_user ? status_user : c->status_dev;
    const bool relabel = n >= kRelabelMinN;
    if (c->graphs && !c->timing && n > 0 && (sparse ? !sparse_waits(c, k, n, m, relabel, 1) : c->state_clean)) {
        // repeat counts replay one CUDA graph of the whole launch sequence;
        // it is captured (on the context's stream, not run) at the second
        // count with the same key, and only while the pair-state buffer is
        // known clean, so it holds no full sweep
        acc_ctx::CountKey key;
        memset(&key, 0, sizeof(key));
        key.rowptr = rowptr;
        key.col = col;
        key.counts = counts;
        key.status = status;
        key.m = m;
        key.light = c->sched_light;
        key.target = c->sched_target;
        key.partial_end = c->partial_arcs_end;
        key.sparse_any = c->sparse_any;
        key.n = n;
        key.k = k;
        key.mode = c->mode;
        key.grid_num = c->grid_num;
        key.grid_den = c->grid_den;
        key.adjacency = c->adjacency;
        const void *ws[32] = {c->state, c->deg, c->lo, c->label, c->deg_in, c->nptr, c->tiles, c->nbr, c->occ,
                              c->info, c->queue, c->scratch, c->lut[k], c->lut_sv[k], c->class_code_dev[k],
                              c->f5_pre, c->status_dev, c->src, c->nh, c->rev, c->pp_nd, c->pp_tri, c->pp_part,
                              c->pp_wedges, c->pp_done, c->p5_vert, c->p5_sums, c->tab5, c->sp_raw, c->sp_merged, c->sp_roff, c->sp_big};
        memcpy(key.ws, ws, sizeof(ws));
        bool have = c->cg_exec && memcmp(&key, &c->cg_key, sizeof(key)) == 0;
        // capture only when a count repeats: a one-off count runs one by one
        const bool repeat = memcmp(&key, &c->cg_seen, sizeof(key)) == 0;
        if (!have && !repeat) c->cg_seen = key;
        if (!have && repeat) {
            if (c->cg_exec) cudaGraphExecDestroy(c->cg_exec);
            c->cg_exec = nullptr;
            cudaGraph_t g = nullptr;
            if (ok(cudaStreamBeginCapture(c->own, cudaStreamCaptureModeRelaxed))) {
                rc = run_set(c, gs, n, k, relabel, c->own, counts, status);
                const cudaError_t ce = cudaStreamEndCapture(c->own, &g);
                if (!sparse) c->state_clean = true;  // nothing ran
                if (rc) {
                    if (g) cudaGraphDestroy(g);
                    return rc;
                }
                if (ce == cudaSuccess && g && ok(cudaGraphInstantiate(&c->cg_exec, g, 0))) {
                    c->cg_key = key;
                    c->cg_launches = c->last_launches;
                    c->cg_partial5 = c->last_partial5;
                    c->cg_units = c->last_units;
                    c->cg_blocks = c->last_blocks;
                    have = true;
                } else {
                    c->cg_exec = nullptr;
                }
                if (g) cudaGraphDestroy(g);
            }
            cudaGetLastError();  // a refused capture leaves the eager path below
        }
        if (have) {
            if (!ok(cudaGraphLaunch(c->cg_exec, s))) return ACC_ERR_CUDA;
            if (!sparse) c->state_clean = true;  // the sequence ends with the clear
            c->last_launches = c->cg_launches;
            c->last_partial5 = c->cg_partial5;
            c->last_k = k;
            c->last_units = c->cg_units;
            c->last_blocks = c->cg_blocks;
            return finish(c, s, status_user);
        }
    }
    rc = run_set(c, gs, n, k, relabel, s, counts, status);
    if (rc) return rc;
    return finish(c, s, status_user);
}

// The workspace a run of the prepared batch needs under the context's
// current mode and adjacency choice, which may differ from those at the
// prepare (the count mode's reverse positions, hashed tables or sparse
// build): grows nothing when they are the same.
int batch_workspace(acc_ctx *c, cudaStream_t s) {
    if (size_check(c, c->batch_max_n)) return ACC_ERR_TOO_LARGE;
    return ensure_workspace(c, c->batch_set.NV, c->batch_words, c->batch_arcs, c->batch_max_n, c->batch_k,
                            c->batch_set.B, true, s);
}

}  // namespace

namespace acc {

long long ctx_footprint(acc_ctx *c, long long n, long long m, int k0, int k1, Ways ways) {
    const long long pitch = state_pitch((int)n), arcs_end = c->partial_arcs_end;
    const bool relabel = n >= kRelabelMinN;
    ctx_allow_partial(c, ways != Ways::kScan);
    // what the context holds already
    long long held = (long long)kQueueCap * 16, least = 0;
    workspace_buffers(c, [&](auto **p, size_t *cap) { held += (long long)(*cap * sizeof(**p)); });
    // what would grow, by the buffer's capacity (workspace_needs names 25)
    struct {
        const size_t *cap;
        long long more;
    } growth[32] = {};
    auto grows = [&](const size_t *cap, size_t need, size_t bytes) {
        if (need <= *cap) return;
        const long long more = (long long)((need + need / 4 + 64 - *cap) * bytes);
        for (auto &g : growth)
            if (!g.cap || g.cap == cap) {
                g.cap = cap;
                g.more = g.more > more ? g.more : more;
                return;
            }
    };
    for (int k = k0; k <= k1; k++) {
        const long long warps = enum_grid_warps(k, c->num_sms) > 0 ? enum_grid_warps(k, c->num_sms) : 0;
        // the list scan's share, whichever way the graph is counted, so that admission
        // does not depend on it.  The sparse build keeps raw and merged rows (2 m words
        // each) and row offsets instead of the dense block and its bitmap; its overflow
        // lists are bounded by the largest degree, itself at most 2m and n
        const bool sparse = sparse_build(c, (int)n);
        const long long hash_bytes = uses_hash(c, k, (int)n) ? 4LL * kNhWords * (2 * m + 1) : 0;
        const long long list_n = sparse ? (2 * m < n ? 2 * m : n) : n;
        const long long lists =
            (sparse ? 2 * sparse_list_entries((int)list_n) + 2 * kPartBRows : scratch_per_warp((int)n)) * warps;
        const long long scan = (sparse ? 16 * (m + 1) + 8 * (n + 1) : n * pitch * 4 + 4 * n * occ_words((int)n)) +
                               5 * 4 * (n + 1) + 8 * (n + 1) + (uses_rev(c, m) ? 16 : 8) * (2 * m + 1) + hash_bytes +
                               (long long)kQueueCap * 16 + lists * 4;
        least = least > scan + scan / 4 ? least : scan + scan / 4;
        workspace_needs(c, n, n * pitch, m, (int)n, k, 1, relabel, (int)warps, ways == Ways::kEither,
                        [&](auto **p, size_t *cap, size_t need) { grows(cap, need, sizeof(**p)); });
        if (sparse_path(c, k, (int)n, m, relabel, 1) && sparse_waits(c, k, (int)n, m, relabel, 1))
            grows(&c->scratch_cap, (size_t)lists, sizeof(*c->scratch));
    }
    c->partial_arcs_end = arcs_end;
    for (const auto &g : growth) held += g.more;
    return held > least ? held : least;
}

int ctx_reserve(acc_ctx *c, long long n, long long m, int k, Ways ways) {
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    const int rc = ensure_tab5(c, c->own);
    if (rc) return rc;
    const bool relabel = n >= kRelabelMinN;
    ctx_allow_partial(c, ways != Ways::kScan);
    return ensure_workspace(c, n, n * state_pitch((int)n), m, (int)n, k, 1, relabel, c->own, ways == Ways::kEither);
}

}  // namespace acc

extern "C" {

const char *acc_strerror(int code) {
    switch (code) {
    case ACC_OK: return "ok";
    case ACC_ERR_K: return "k must be 3, 4 or 5";
    case ACC_ERR_INPUT: return "malformed graph (rowptr, column range, self-loop or size)";
    case ACC_ERR_NOMEM: return "device or pinned-host allocation failed";
    case ACC_ERR_TIMEOUT: return "a bounded device wait gave up";
    case ACC_ERR_OVERFLOW: return "a count or an index would not fit its type";
    case ACC_ERR_CUDA: return "a CUDA runtime call failed";
    case ACC_ERR_ARG: return "null pointer, bad handle or bad option";
    case ACC_ERR_TOO_LARGE: return "n above ACC_MAX_N (ACC_MAX_N_SPARSE in the count mode)";
    case ACC_ERR_INTERNAL: return "internal consistency check failed";
    default: return "unknown error";
    }
}

int acc_motif_num_classes(int k) { return valid_k(k) ? num_classes(k) : ACC_ERR_K; }

int acc_ctx_create(acc_ctx **out, int device) {
    if (!out) return ACC_ERR_ARG;
    *out = nullptr;
    acc_ctx *c = new (std::nothrow) acc_ctx();
    if (!c) return ACC_ERR_NOMEM;
    c->device = device;
    if (!set_device(device) ||
        !ok(cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device)) ||
        !ok(cudaStreamCreateWithFlags(&c->own, cudaStreamNonBlocking)) ||
        !ok(cudaMallocHost(&c->status_host, sizeof(int)))) {
        cudaGetLastError();
        acc_ctx_destroy(c);
        return ACC_ERR_CUDA;
    }
    *out = c;
    return ACC_OK;
}

void acc_ctx_destroy(acc_ctx *c) {
    if (!c) return;
    cudaSetDevice(c->device);
    cudaDeviceSynchronize();
    release_luts(c);
    cudaFree(c->state);
    cudaFree(c->deg);
    cudaFree(c->lo);
    cudaFree(c->nptr);
    cudaFree(c->label);
    cudaFree(c->deg_in);
    cudaFree(c->tiles);
    cudaFree(c->f5_pre);
    cudaFree(c->occ);
    cudaFree(c->nbr);
    cudaFree(c->src);
    cudaFree(c->rev);
    cudaFree(c->nh);
    cudaFree(c->pp_nd);
    cudaFree(c->pp_tri);
    cudaFree(c->pp_part);
    cudaFree(c->pp_wedges);
    cudaFree(c->pp_done);
    cudaFree(c->p5_vert);
    cudaFree(c->p5_sums);
    cudaFree(c->sp_raw);
    cudaFree(c->sp_merged);
    cudaFree(c->sp_roff);
    cudaFree(c->sp_big);
    if (c->maxdeg_host) cudaFreeHost(c->maxdeg_host);
    cudaFree(c->info);
    cudaFree(c->queue);
    cudaFree(c->scratch);
    cudaFree(c->status_dev);
    cudaFree(c->meta_dev);
    cudaFree(c->gid);
    if (c->cg_exec) cudaGraphExecDestroy(c->cg_exec);
    cudaFree(c->rand_meta);
    cudaFree(c->rand_rows);
    cudaFree(c->rand_bits);
    cudaFree(c->rand_rpart);
    cudaFree(c->rand_pts);
    cudaFree(c->h2d_rowptr);
    cudaFree(c->h2d_col);
    cudaFree(c->h2d_counts);
    for (int i = 0; i < 4; i++)
        if (c->ev[i]) cudaEventDestroy(c->ev[i]);
    if (c->status_host) cudaFreeHost(c->status_host);
    if (c->own) cudaStreamDestroy(c->own);
    cudaGetLastError();
    delete c;
}

int acc_motif_prepare(acc_ctx *c, int k, void *stream) {
    if (!c) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    c->partial_arcs_end = INT64_MAX;
    c->sparse_any = false;
    int rc = k == 5 ? ensure_tab5(c, s) : ensure_lut(c, k, s);
    if (rc) return rc;
    return ok(cudaStreamSynchronize(s)) ? ACC_OK : ACC_ERR_CUDA;
}

int acc_motif_count(acc_ctx *c, const int64_t *d_rowptr, const int32_t *d_col, int32_t n, int64_t m, int k,
                    void *stream, int64_t *d_counts, int32_t *d_status) {
    return count_impl(c, d_rowptr, d_col, n, m, k, (cudaStream_t)stream, d_counts, d_status);
}

int acc_motif_count_host(acc_ctx *c, const int64_t *h_rowptr, const int32_t *h_col, int32_t n, int64_t m, int k,
                         int64_t *h_counts) {
    if (!c || !h_rowptr || !h_counts || (m > 0 && !h_col)) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (n < 0 || m < 0 || m >= (1ll << 31)) return ACC_ERR_INPUT;
    if (size_check(c, n)) return ACC_ERR_TOO_LARGE;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    int rc;
    size_t cnt_cap = c->h2d_counts ? 9364 : 0;
    if ((rc = grow(&c->h2d_rowptr, &c->h2d_rowptr_cap, (size_t)n + 1))) return rc;
    if ((rc = grow(&c->h2d_col, &c->h2d_col_cap, (size_t)m + 1))) return rc;
    if ((rc = grow(&c->h2d_counts, &cnt_cap, 9364))) return rc;
    cudaStream_t s = c->own;
    if (!ok(cudaMemcpyAsync(c->h2d_rowptr, h_rowptr, ((size_t)n + 1) * 8, cudaMemcpyHostToDevice, s)))
        return ACC_ERR_CUDA;
    if (m > 0 && !ok(cudaMemcpyAsync(c->h2d_col, h_col, (size_t)m * 4, cudaMemcpyHostToDevice, s)))
        return ACC_ERR_CUDA;
    rc = count_impl(c, reinterpret_cast<const int64_t *>(c->h2d_rowptr), c->h2d_col, n, m, k, s,
                    reinterpret_cast<int64_t *>(c->h2d_counts), c->status_dev);
    if (rc) return rc;
    if (!ok(cudaMemcpyAsync(h_counts, c->h2d_counts, (size_t)num_classes(k) * 8, cudaMemcpyDeviceToHost, s)))
        return ACC_ERR_CUDA;
    if (!ok(cudaMemcpyAsync(c->status_host, c->status_dev, sizeof(int), cudaMemcpyDeviceToHost, s)))
        return ACC_ERR_CUDA;
    if (!ok(cudaStreamSynchronize(s))) return ACC_ERR_CUDA;
    return *c->status_host;
}

int acc_motif_batch_prepare(acc_ctx *c, const acc_graph_desc *graphs, int32_t B, int k, void *stream) {
    if (!c || (B > 0 && !graphs) || B < 0) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    c->batch_ready = false;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<GMeta> metas((size_t)B);
    long long NV = 0, words = 0, arcs = 0;
    int max_n = 0;
    for (int g = 0; g < B; g++) {
        const acc_graph_desc &d = graphs[g];
        if (!d.rowptr || (d.m > 0 && !d.col)) return ACC_ERR_ARG;
        if (d.n < 0 || d.m < 0 || d.m >= (1ll << 31)) return ACC_ERR_INPUT;
        if (size_check(c, d.n)) return ACC_ERR_TOO_LARGE;
        GMeta &mt = metas[(size_t)g];
        mt.rowptr = reinterpret_cast<const long long *>(d.rowptr);
        mt.col = d.col;
        mt.m = d.m;
        mt.n = d.n;
        mt.pitch = state_pitch(d.n);
        mt.soff = words;
        mt.moff = arcs;
        mt.voff = (int)NV;
        words += (long long)d.n * mt.pitch;
        NV += d.n;
        arcs += d.m;
        if (d.n > max_n) max_n = d.n;
        if (NV >= (1ll << 31) || arcs >= (1ll << 31)) return ACC_ERR_OVERFLOW;
    }
    // an earlier run on this stream (enqueued only, when it had a status
    // word) may still read the descriptors and graph ids rewritten below;
    // the pageable copy would not wait for it
    if (!ok(cudaStreamSynchronize(s))) return ACC_ERR_CUDA;
    // (k = 5: also for a run after the mode changed to the count mode)
    int rc = k == 5 && B == 1 ? ensure_tab5(c, s) : ensure_lut(c, k, s);
    if (rc) return rc;
    c->partial_arcs_end = INT64_MAX;
    c->sparse_any = false;
    if ((rc = ensure_workspace(c, NV, words, arcs, max_n, k, B, true, s))) return rc;
    if ((rc = grow(&c->meta_dev, &c->meta_cap, (size_t)B + 1))) return rc;
    if ((rc = grow(&c->gid, &c->gid_cap, (size_t)NV + 1))) return rc;
    // (copies from pageable memory return when staged: on the stream that reads them,
    // which need not wait for the legacy stream)
    if (B > 0 &&
        !ok(cudaMemcpyAsync(c->meta_dev, metas.data(), sizeof(GMeta) * (size_t)B, cudaMemcpyHostToDevice, s)))
        return ACC_ERR_CUDA;
    GSet gs = {};
    if (B == 1) gs.one = metas[0];
    gs.many = c->meta_dev;
    gs.gid = c->gid;
    gs.B = B;
    gs.NV = NV;
    gs.M = arcs;
    if ((rc = launch_graph_ids(gs, c->gid, s)) < 0) return rc;
    if (!ok(cudaStreamSynchronize(s))) return ACC_ERR_CUDA;
    c->batch_set = gs;
    c->batch_k = k;
    c->batch_words = words;
    c->batch_arcs = arcs;
    c->batch_max_n = max_n;
    c->batch_ready = true;
    return ACC_OK;
}

int acc_motif_batch_run(acc_ctx *c, void *stream, int64_t *d_counts, int32_t *d_status) {
    if (!c || !d_counts || !c->batch_ready) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    if (c->batch_set.B == 0) return ACC_OK;
    int rc = batch_workspace(c, s);
    if (rc) return rc;
    int *status = d_status ? d_status : c->status_dev;
    rc = run_set(c, c->batch_set, c->batch_max_n, c->batch_k, true, s, d_counts, status);
    if (rc) return rc;
    return finish(c, s, d_status);
}

int acc_motif_count_batch(acc_ctx *c, const acc_graph_desc *graphs, int32_t B, int k, void *stream,
                          int64_t *d_counts, int32_t *d_status) {
    const int rc = acc_motif_batch_prepare(c, graphs, B, k, stream);
    if (rc) return rc;
    return acc_motif_batch_run(c, stream, d_counts, d_status);
}

int acc_motif_zscores(const int64_t *d_counts, int32_t groups, int32_t group_size, int k, void *stream,
                      double *d_z) {
    if (!valid_k(k)) return ACC_ERR_K;
    if (groups < 0 || group_size < 2) return ACC_ERR_ARG;
    if (groups > 0 && (!d_counts || !d_z)) return ACC_ERR_ARG;
    const int rc = launch_zscores(reinterpret_cast<const long long *>(d_counts), groups, group_size, num_classes(k),
                                  d_z, (cudaStream_t)stream);
    return rc < 0 ? rc : ACC_OK;
}

int acc_swap_randomise(acc_ctx *c, const acc_graph_desc *graphs, int32_t G, int32_t R, int64_t attempts_per_arc,
                       const uint64_t *seeds, int mode, void *stream, int32_t *d_out, int64_t *d_accepted,
                       int32_t *d_status) {
    if (!c || G < 0 || R < 0 || attempts_per_arc < 0) return ACC_ERR_ARG;
    if (mode != ACC_RAND_SWAP && mode != ACC_RAND_MUTUAL) return ACC_ERR_ARG;
    if (G > 0 && (!graphs || !seeds)) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<RGraph> metas((size_t)G);
    long long M = 0, NV = 0, bwords = 0;
    for (int g = 0; g < G; g++) {
        const acc_graph_desc &d = graphs[g];
        if (!d.rowptr || (d.m > 0 && !d.col)) return ACC_ERR_ARG;
        if (d.n < 0 || d.m < 0 || d.m >= (1ll << 31) || (d.n == 0 && d.m > 0)) return ACC_ERR_INPUT;
        if (d.m > 0 && attempts_per_arc > (1ll << 62) / d.m) return ACC_ERR_OVERFLOW;
        RGraph &rg = metas[(size_t)g];
        rg.rowptr = reinterpret_cast<const long long *>(d.rowptr);
        rg.col = d.col;
        rg.m = d.m;
        rg.n = d.n;
        rg.moff = M;
        rg.ooff = M * (long long)R;
        rg.attempts = attempts_per_arc * d.m;
        rg.seed = seeds[g];
        rg.voff = (int)NV;
        rg.bw = (int)((((long long)d.n + 31) / 32 + 3) & ~3ll);
        rg.boff = bwords;
        M += d.m;
        NV += d.n;
        if (M >= (1ll << 40) || NV >= (1ll << 31)) return ACC_ERR_OVERFLOW;
        const long long per_copy = (long long)d.n * rg.bw;
        bwords = (R > 0 && per_copy > ((1ll << 60) - bwords) / R) ? (1ll << 60) : bwords + per_copy * R;
    }
    if (R > 0 && M > (1ll << 62) / R) return ACC_ERR_OVERFLOW;
    if (M * (long long)R > 0 && !d_out) return ACC_ERR_ARG;
    int rc;
    const bool same = c->rand_meta && c->rand_rows && c->rand_host.size() == metas.size() &&
                      (G == 0 || memcmp(c->rand_host.data(), metas.data(), sizeof(RGraph) * (size_t)G) == 0);
    if (!same) {
        // the previous call on this stream may still read the descriptors
        if (!ok(cudaStreamSynchronize(s))) return ACC_ERR_CUDA;
        c->rand_host.clear();
        if ((rc = grow(&c->rand_meta, &c->rand_meta_cap, (size_t)G + 1))) return rc;
        if ((rc = grow(&c->rand_rows, &c->rand_rows_cap, (size_t)M + 1))) return rc;
        if (G > 0 &&
            !ok(cudaMemcpyAsync(c->rand_meta, metas.data(), sizeof(RGraph) * (size_t)G, cudaMemcpyHostToDevice, s)))
            return ACC_ERR_CUDA;
        c->rand_host = metas;
    }
    // both modes run speculatively when the copies' adjacency bitmaps (and,
    // for the mutual mode, the reverse positions of the graphs' and the
    // copies' arcs) fit the limit, and half of the free device memory when
    // they must grow
    uint32_t *bits = nullptr;
    int *rpart = nullptr, *pts = nullptr;
    const bool mutual = mode == ACC_RAND_MUTUAL;
    const long long extra = mutual ? M + M * (long long)R : 0;  // ints
    if (bwords > 0 && bwords < (1ll << 60) && (bwords + extra) * 4 <= c->rand_bits_limit) {
        bool fits = (size_t)bwords <= c->rand_bits_cap &&
                    (!mutual || ((size_t)M <= c->rand_rpart_cap && (size_t)(M * (long long)R) <= c->rand_pts_cap));
        if (!fits) {
            size_t free_b = 0, total_b = 0;
            fits = ok(cudaMemGetInfo(&free_b, &total_b)) && (size_t)(bwords + extra) * 4 * 2 <= free_b;
            cudaGetLastError();
            if (fits && grow(&c->rand_bits, &c->rand_bits_cap, (size_t)bwords) != ACC_OK) fits = false;
            if (fits && mutual &&
                (grow(&c->rand_rpart, &c->rand_rpart_cap, (size_t)M) != ACC_OK ||
                 grow(&c->rand_pts, &c->rand_pts_cap, (size_t)(M * (long long)R)) != ACC_OK))
                fits = false;
        }
        if (fits) {
            bits = c->rand_bits;
            if (mutual) {
                rpart = c->rand_rpart;
                pts = c->rand_pts;
            }
        }
    }
    if (!c->status_dev && !ok(cudaMalloc(&c->status_dev, sizeof(int)))) return ACC_ERR_NOMEM;
    int *status = d_status ? d_status : c->status_dev;
    if (!ok(cudaMemsetAsync(status, 0, sizeof(int), s))) return ACC_ERR_CUDA;
    rc = launch_randomise(c->rand_meta, G, R, M, NV, mode, c->rand_rows, d_out, bits, rpart, pts,
                          reinterpret_cast<long long *>(d_accepted), status, c->num_sms, s);
    if (rc < 0) return rc;
    return finish(c, s, d_status);
}

int acc_ctx_set_launch_graphs(acc_ctx *c, int on) {
    if (!c || (on != 0 && on != 1)) return ACC_ERR_ARG;
    c->graphs = on != 0;
    return ACC_OK;
}

int acc_ctx_set_randomise_memory(acc_ctx *c, int64_t bytes) {
    if (!c || bytes < 0) return ACC_ERR_ARG;
    c->rand_bits_limit = bytes;
    return ACC_OK;
}

int acc_motif_class_code(acc_ctx *c, int k, int32_t cls, uint32_t *code) {
    if (!c || !code) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (cls < 0 || cls >= num_classes(k)) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    int rc = ensure_lut(c, k, c->own);
    if (rc) return rc;
    *code = c->class_code_host[k][cls];
    return ACC_OK;
}

int acc_motif_classify_code(acc_ctx *c, int k, uint32_t code, int32_t *cls) {
    if (!c || !cls) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (code >= (1u << code_bits(k))) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    int rc = ensure_lut(c, k, c->own);
    if (rc) return rc;
    *cls = c->lut_host[k][code];
    return ACC_OK;
}

int acc_motif_copy_table(acc_ctx *c, int k, int16_t *h_table) {
    if (!c || !h_table) return ACC_ERR_ARG;
    if (!valid_k(k)) return ACC_ERR_K;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    int rc = ensure_lut(c, k, c->own);
    if (rc) return rc;
    memcpy(h_table, c->lut_host[k], (size_t(1) << code_bits(k)) * 2);
    return ACC_OK;
}

int acc_motif_last_stats(acc_ctx *c, int64_t *h_stats) {
    if (!c || !h_stats) return ACC_ERR_ARG;
    if (!c->info) return ACC_ERR_ARG;
    if (!set_device(c->device) || !ok(cudaDeviceSynchronize())) return ACC_ERR_CUDA;
    GraphInfo gi;
    if (!ok(cudaMemcpy(&gi, c->info, sizeof(gi), cudaMemcpyDeviceToHost))) return ACC_ERR_CUDA;
    h_stats[0] = c->last_launches;
    h_stats[1] = c->last_k == 3 ? (int64_t)c->last_units : (int64_t)gi.nnz;
    h_stats[2] = (int64_t)gi.queue_tail;
    if (c->last_partial5 && c->p5_sums) {
        unsigned long long ctr[kCtrs];
        if (!ok(cudaMemcpy(ctr, c->p5_sums + num_classes(5) + 16, sizeof(ctr), cudaMemcpyDeviceToHost))) return ACC_ERR_CUDA;
        h_stats[2] += (int64_t)(ctr[kCtrPairTail] + ctr[kCtrTail4] + ctr[kCtrCycTail]);
    }
    h_stats[3] = (int64_t)(gi.nnz / 2);
    h_stats[4] = gi.maxdeg;
    h_stats[5] = c->last_blocks;
    h_stats[6] = (int64_t)gi.scanned;
    return ACC_OK;
}

int acc_ctx_set_adjacency(acc_ctx *c, int adjacency) {
    if (!c || (adjacency != ACC_ADJ_AUTO && adjacency != ACC_ADJ_DENSE && adjacency != ACC_ADJ_HASH &&
               adjacency != ACC_ADJ_SPARSE))
        return ACC_ERR_ARG;
    c->adjacency = adjacency;
    return ACC_OK;
}

int acc_ctx_set_mode(acc_ctx *c, int mode) {
    if (!c || (mode != ACC_MODE_COUNT && mode != ACC_MODE_ENUMERATE && mode != ACC_MODE_FORMULA &&
               mode != ACC_MODE_AUTO))
        return ACC_ERR_ARG;
    c->mode = mode;
    return ACC_OK;
}

int acc_ctx_set_schedule(acc_ctx *c, int64_t light, int64_t target) {
    constexpr int64_t kMax = 1ll << 40;
    if (!c || light < 0 || target < 0 || light > kMax || target > kMax) return ACC_ERR_ARG;
    c->sched_light = light;
    c->sched_target = target;
    return ACC_OK;
}

int acc_ctx_get_schedule(acc_ctx *c, int64_t *light, int64_t *target) {
    if (!c || !light || !target) return ACC_ERR_ARG;
    *light = c->sched_light > 0 ? c->sched_light : enum_default_light(3, true);
    *target = c->sched_target > 0 ? c->sched_target : enum_default_target(3, true);
    return ACC_OK;
}

int acc_motif_batch_autotune(acc_ctx *c, void *stream, int64_t *h_light, int64_t *h_target, float *h_ms) {
    if (!c || !c->batch_ready) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const long long B = c->batch_set.B;
    const long long light0 = c->sched_light, target0 = c->sched_target;
    // candidate schedules: light units from a warp each up to large units,
    // heavy units cut into small or large row tiles
    const long long lights[] = {512, 2048, 8192, 32768, 131072, 1ll << 20};
    const long long targets[] = {1024, 4096, 16384};
    int64_t *counts = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = ACC_OK;
    long long best_l = 0, best_t = 0;
    float best = -1.0f;
    auto timed_run = [&](float *ms) -> int {
        if (!ok(cudaEventRecord(e0, s))) return ACC_ERR_CUDA;
        const int r = run_set(c, c->batch_set, c->batch_max_n, c->batch_k, true, s, counts, c->status_dev);
        if (r) return r;
        if (!ok(cudaEventRecord(e1, s)) || !ok(cudaEventSynchronize(e1)) || !ok(cudaEventElapsedTime(ms, e0, e1)))
            return ACC_ERR_CUDA;
        return finish(c, s, nullptr);  // a failing batch fails the tuning
    };
    const bool partial5 = uses_partial5(c, c->batch_k, c->batch_max_n, c->batch_arcs, true, (int)B);
    bool scans = !uses_formula(c, c->batch_k, c->batch_max_n) &&
                 !uses_partial(c, c->batch_k, c->batch_max_n, c->batch_arcs, true, (int)B);
    if (B == 0) {
        best_l = enum_default_light(c->batch_k, c->mode != ACC_MODE_ENUMERATE);
        best_t = enum_default_target(c->batch_k, c->mode != ACC_MODE_ENUMERATE);
        best = 0.0f;
        goto done;
    }
    if ((rc = batch_workspace(c, s))) return rc;
    if (!ok(cudaMalloc(&counts, (size_t)B * num_classes(c->batch_k) * sizeof(int64_t)))) return ACC_ERR_NOMEM;
    if (!ok(cudaEventCreate(&e0)) || !ok(cudaEventCreate(&e1))) {
        rc = ACC_ERR_CUDA;
        goto done;
    }
    // A batch that no scan counts does not read the schedule: its runs differ by
    // noise alone, and the luckiest pair would be kept for the context's next
    // scans.  Timed (the second run), the schedule kept as it was.
    for (int rep = 0; rep < 2 && (!scans || partial5); rep++) {
        if ((rc = timed_run(&best))) goto done;
        if (partial5 && rep == 0) {
            unsigned long long scan = 0;
            if (!ok(cudaMemcpy(&scan, c->p5_sums + num_classes(5) + 16 + kCtrScan, sizeof(scan), cudaMemcpyDeviceToHost))) {
                rc = ACC_ERR_CUDA;
                goto done;
            }
            scans = scan != 0;
            if (scans) break;
        }
    }
    if (!scans) {
        best_l = light0;
        best_t = target0;
        goto done;
    }
    best = -1.0f;
    for (long long l : lights) {
        for (long long t : targets) {
            c->sched_light = l;
            c->sched_target = t;
            float ms = 0.0f;
            if ((rc = timed_run(&ms))) goto done;
            if (best < 0.0f || ms < best) {
                best = ms;
                best_l = l;
                best_t = t;
            }
        }
    }
done:
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(counts);
    if (rc) {
        c->sched_light = light0;
        c->sched_target = target0;
        return rc;
    }
    c->sched_light = best_l;
    c->sched_target = best_t;
    int64_t light, target;
    acc_ctx_get_schedule(c, &light, &target);
    if (h_light) *h_light = light;
    if (h_target) *h_target = target;
    if (h_ms) *h_ms = best;
    return ACC_OK;
}

int acc_ctx_set_timing(acc_ctx *c, int on) {
    if (!c) return ACC_ERR_ARG;
    if (!set_device(c->device)) return ACC_ERR_CUDA;
    if (on && !c->ev[0]) {
        for (int i = 0; i < 4; i++)
            if (!ok(cudaEventCreate(&c->ev[i]))) {
                cudaGetLastError();
                return ACC_ERR_CUDA;
            }
    }
    c->timing = on != 0;
    return ACC_OK;
}

int acc_motif_last_timing(acc_ctx *c, float *h_ms) {
    if (!c || !h_ms || !c->timed_call) return ACC_ERR_ARG;
    if (!set_device(c->device) || !ok(cudaEventSynchronize(c->ev[2]))) return ACC_ERR_CUDA;
    if (!ok(cudaEventElapsedTime(&h_ms[0], c->ev[0], c->ev[1])) ||
        !ok(cudaEventElapsedTime(&h_ms[1], c->ev[1], c->ev[2])) ||
        !ok(cudaEventElapsedTime(&h_ms[2], c->ev[1], c->ev[3])) ||
        !ok(cudaEventElapsedTime(&h_ms[3], c->ev[3], c->ev[2])))
        return ACC_ERR_CUDA;
    return ACC_OK;
}

}  // extern "C"
