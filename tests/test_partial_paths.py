"""The ways a count by partial patterns (csrc/partial.cu, csrc/partial5.cu) can
take besides the common one, on the host: the library's own source runs there
(tests/emu) with the size threshold at 0, against the oracle.

The graphs that take these ways in earnest are too large for the host, so the
sources' limits are read from the environment where EDITS puts emu_env (their
own value where the variable is not set), and k_cycles5 can be told to find the
return to the list scan raised while the warps of its first block start."""
import ctypes
import json
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import oracle
from tests.graph_helpers import random_digraph
from tests.test_partial import fan

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

HOOKS = r"""
#include "shim.h"
inline unsigned long long emu_env(const char *name, unsigned long long own) {
    const char *e = getenv(name);
    return e ? strtoull(e, nullptr, 10) : own;
}
// device memory: bytes held, and the most that may be
extern unsigned long long emu_held, emu_most;
std::map<void *, size_t> &emu_sizes();
template <class T> inline cudaError_t emu_counted_malloc(T **p, size_t bytes) {
    if (emu_held + bytes > emu_most) {
        *p = nullptr;
        return 2;  // out of memory
    }
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaSuccess) emu_held += emu_sizes()[*p] = bytes;
    return e;
}
template <class T> inline cudaError_t emu_counted_free(T *p) {
    auto it = emu_sizes().find((void *)p);
    if (it != emu_sizes().end()) {
        emu_held -= it->second;
        emu_sizes().erase(it);
    }
    return cudaFree((void *)p);
}
// two devices; a kernel's limit of shared memory is set on the current one
extern int emu_device;
void emu_limit_set(const void *kernel, int bytes);
inline cudaError_t emu_set_device(int d) {
    if (d < 0 || d > 1) return 1;
    emu_device = d;
    return cudaSuccess;
}
inline cudaError_t emu_get_device(int *d) {
    *d = emu_device;
    return cudaSuccess;
}
template <class T> inline cudaError_t emu_set_limit(T kernel, cudaFuncAttribute, int bytes) {
    emu_limit_set((const void *)kernel, bytes);
    return cudaSuccess;
}
// deferred mode (EMU_DEFER=1): a copy from pageable memory and a set return before
// they are done, and a stream of its own does not wait for the legacy stream
inline cudaError_t emu_late_memcpy(void *d, const void *s, size_t n, cudaMemcpyKind kind) {
    if (kind != cudaMemcpyHostToDevice || !emu_defer() || emu_is_pinned(s)) return cudaMemcpy(d, s, n, kind);
    emu_flush(nullptr);
    std::vector<char> staged((const char *)s, (const char *)s + n);
    emu_submit(nullptr, [=] { memcpy(d, staged.data(), n); });
    return cudaSuccess;
}
inline cudaError_t emu_late_memset(void *d, int v, size_t n) {
    emu_submit(nullptr, [=] { memset(d, v, n); });
    return cudaSuccess;
}
#define cudaMemcpy emu_late_memcpy
#define cudaMemset emu_late_memset
#define cudaSetDevice emu_set_device
#define cudaGetDevice emu_get_device
#define cudaFuncSetAttribute emu_set_limit
#define cudaMalloc emu_counted_malloc
#define cudaFree emu_counted_free
extern unsigned long long emu_scans;  // k = 5 counts left to the list scan
extern unsigned long long emu_partials;  // k = 3, 4 sets counted by partial patterns
// k_cycles5<phase>: what other blocks left in shared memory, as the first thread
// of a block finds it, and the flag raised when thread EMU_RAISE_AT of the first block
// arrives
template <class A> inline void emu_cycles_enter(const A &a, unsigned long long *flag, int phase, size_t smem) {
    static unsigned entered = 0;
    if (emu_env("EMU_RAISE_PHASE", 0) != (unsigned long long)phase) return;
    if (entered % blockDim.x == 0) memset(emu_dyn_smem, 0xA5, smem);
    if (entered++ < blockDim.x && threadIdx.x == emu_env("EMU_RAISE_AT", 0)) *flag = 1;
}
"""

GLOBALS = r"""
#include "hooks.h"
#include "context.cuh"
extern "C" long long emu_footprint(acc_ctx *c, long long n, long long m, int k0, int k1, int ways) {
    return acc::ctx_footprint(c, n, m, k0, k1, (acc::Ways)ways);
}
extern "C" int emu_reserve(acc_ctx *c, long long n, long long m, int k, int ways) {
    return acc::ctx_reserve(c, n, m, k, (acc::Ways)ways);
}
unsigned long long emu_scans = 0, emu_partials = 0, emu_held = 0, emu_most = ~0ull;
std::map<void *, size_t> &emu_sizes() {
    static std::map<void *, size_t> m;
    return m;
}
int emu_device = 0;
static std::map<const void *, int> emu_limits[2];
void emu_limit_set(const void *kernel, int bytes) { emu_limits[emu_device][kernel] = bytes; }
// kernels whose limit was raised on device 0, and on both devices alike
extern "C" void emu_limit_counts(int *first, int *both) {
    *first = (int)emu_limits[0].size();
    *both = 0;
    for (auto &l : emu_limits[0]) *both += emu_limits[1].count(l.first) && emu_limits[1][l.first] == l.second;
}
extern "C" unsigned long long emu_scan_count() { return emu_scans; }
extern "C" unsigned long long emu_partial_count() { return emu_partials; }
extern "C" unsigned long long emu_bytes() { return emu_held; }
extern "C" void emu_limit(unsigned long long most) { emu_most = most; }
"""

# (source file, text in it, what stands there for these tests)
EDITS = [
    ("partial5.cu", "    grid_dep_launch();  // k_wedges<4, PHASE> runs beside\n",
     "    emu_cycles_enter(a, a.p5.ctr + kCtrScan, PHASE, cycle_smem(PHASE));\n"),
    ("partial5.cu", "template <int PHASE>\n__global__ void __launch_bounds__(kCThreads",
     "constexpr size_t cycle_smem(int phase);\ntemplate <int PHASE>\n__global__ void __launch_bounds__(kCThreads"),
    ("api.cu", "(arcs >= 2ll * n || arcs >= ACC_PARTIAL_MIN_ARCS1);",
     "(arcs >= 2ll * n || arcs >= (long long)emu_env(\"EMU_ARCS1\", ACC_PARTIAL_MIN_ARCS1));"),
    ("api.cu", "q.tri_cap = c->scratch_cap / 4;", "q.tri_cap = emu_env(\"EMU_TRIANGLES\", c->scratch_cap / 4);"),
    ("partial.cu", "return d > kFieldMax ?", "return d > (int)emu_env(\"EMU_FIELD\", kFieldMax) ?"),
    ("partial.cu", "const bool wide = rows > kFieldMax;", "const bool wide = rows > (int)emu_env(\"EMU_FIELD\", kFieldMax);"),
    ("partial5.cu", "lo < n && nr < kCRanges", "lo < n && nr < (int)emu_env(\"EMU_RANGES\", kCRanges)"),
    ("partial.cu", "a.info->maxdeg > kCycleRows", "a.info->maxdeg > (int)emu_env(\"EMU_ROWS\", kCycleRows)"),
    ("partial.cu", "- a.lo[v] > kCycleRows", "- a.lo[v] > (int)emu_env(\"EMU_ROWS\", kCycleRows)"),
    ("partial.cu", "    if (k == 3) launch_pdl(k_partial_prep<3>", "    emu_partials++;\n    if (k == 3) launch_pdl(k_partial_prep<3>"),
    ("partial5.cu", "__global__ void __launch_bounds__(256) k_counts5(PartialArgs a) {\n    grid_dep_wait();\n",
     "__global__ void __launch_bounds__(256) k_counts5(PartialArgs a) {\n"
     "    if (threadIdx.x == 0 && blockIdx.x == 0 && a.p5.ctr[kCtrScan]) emu_scans++;\n"),
]


@pytest.fixture(scope="module")
def host_lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from tests.test_cpu_emulation import CSRC, EMU, _launches_to_calls
    out = tmp_path_factory.mktemp("partial_paths")
    units = [os.path.join(EMU, "emu_rt.cpp"), str(out / "hooks.cpp")]
    open(out / "hooks.h", "w").write("#pragma once\n" + HOOKS)
    open(units[1], "w").write(GLOBALS)
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            src = open(os.path.join(CSRC, name)).read()
            for file, text, there in EDITS:
                if file == name:
                    assert src.count(text) == 1, (file, text)
                    src = src.replace(text, there)
            units.append(str(out / (name[:-3] + ".cpp")))
            open(units[-1], "w").write('#include "hooks.h"\n' + _launches_to_calls(src))
    asan = subprocess.run(["g++", "-print-file-name=libasan.so"], capture_output=True, text=True).stdout.strip()
    san = ["-fsanitize=address", "-DEMU_EXACT_ALLOC", "-DEMU_LANE_STACK=65536"] if os.path.isabs(asan) else []
    procs = [subprocess.Popen(["g++", "-std=c++20", "-O1", "-fPIC", "-pthread", "-w", *san, "-DACC_PARTIAL_MIN_ARCS=0", "-DACC_QUEUE_CAP=1024ull", "-DACC_SPARSE_MIN_N=20000", "-DACC_CYCLE_SLOTS=256",
                               "-DEMU_NUM_SMS=1", "-I", str(out), "-I", EMU, "-I", os.path.join(EMU, "fake"), "-I", CSRC,
                               "-c", u, "-o", str(out / f"u{i}.o")], stderr=subprocess.PIPE, text=True)
             for i, u in enumerate(units)]
    for p in procs:
        err = p.communicate()[1]
        assert p.returncode == 0, err[-3000:]
    so = str(out / "lib.so")
    subprocess.run(["g++", "-shared", "-pthread", *san[:1], "-o", so] +
                   [str(out / f"u{i}.o") for i in range(len(units))], check=True)
    return so, dict(os.environ, PYTHONPATH=ROOT, **({"LD_PRELOAD": asan, "ASAN_OPTIONS": "detect_leaks=0"} if san else {}))


# test -> (function host_<name> of this file, environment): each in a process of
# its own, all side by side
RUNS = {}


@pytest.fixture(scope="module")
def on_host(host_lib):
    so, base = host_lib
    procs = {k: subprocess.Popen([sys.executable, os.path.abspath(__file__), so, name], cwd=ROOT,
                                 env=dict(base, **{e: str(v) for e, v in env.items()}), stdout=subprocess.PIPE,
                                 stderr=subprocess.STDOUT, text=True) for k, (name, env) in RUNS.items()}
    yield lambda key: finish(procs[key])
    for p in procs.values():
        p.kill()
        p.wait()


def finish(p):
    """What a process's function returned."""
    out = p.communicate(timeout=300)[0]
    assert p.returncode == 0, out[-3000:]
    return json.loads(out.strip().splitlines()[-1])


# --------------------------------------------------------------------------
# in the process with the host library
# --------------------------------------------------------------------------

def count_set(lib, c, gs, k):
    """Counts of one set (renumbered by degree, whatever its size), status 0."""
    from tests.emu.lib_scenarios import NCLS, P, _descs, ok, sync
    descs, keep = _descs(gs)
    ok(lib.acc_motif_batch_prepare(c.h, descs, len(gs), k, None), "batch_prepare")
    out, st = np.zeros((len(gs), NCLS[k]), np.int64), np.full(1, -1, np.int32)
    ok(lib.acc_motif_batch_run(c.h, None, P(out), P(st)), "batch_run")
    sync(lib)
    assert st[0] == 0, st
    for o, g in zip(out, gs):
        assert np.array_equal(o, oracle.count(*g, k))
    return out


def host_k5_scans(lib):
    """Counts of a k = 5 graph; how often the list scan counted it."""
    from tests.emu.lib_scenarios import Ctx
    c = Ctx(lib)
    count_set(lib, c, [fan(13, 12, 20, 1)], 5)
    c.close()
    return lib.emu_scan_count()


def host_returns(lib):
    """How often the list scan counted: a k = 5 graph of many triangles, one with a
    root of more wedges than a 5-cycle table takes."""
    from tests.emu.lib_scenarios import Ctx
    s, d = random_digraph(np.random.default_rng(9), 14, p=0.4, recip=0.5)
    seen = []
    for g in ((14, np.asarray(s, np.int64), np.asarray(d, np.int64)), fan(40, 6, 150, 1)):
        c = Ctx(lib)
        before = lib.emu_scan_count()
        count_set(lib, c, [g], 5)
        c.close()
        seen.append(lib.emu_scan_count() - before)
    return seen


def host_wide(lib):
    """Sets with roots of more rows than a table's 10-bit fields count (20 of them)."""
    from tests.emu.lib_scenarios import Ctx
    c = Ctx(lib)
    count_set(lib, c, [fan(40, 20, 30, 2), fan(12, 12, 40, 3), fan(60, 30, 900, 3)], 4)
    count_set(lib, c, [fan(40, 20, 30, 2)], 4)
    count_set(lib, c, [fan(22, 9, 20, 1)], 5)
    c.close()
    return lib.emu_scan_count()


def host_k5_parts(lib):
    """Parts of the roots with many wedges of a k = 5 graph, as the statistics have
    them."""
    from tests.emu.lib_scenarios import Ctx, P, ok
    c = Ctx(lib)
    stats = np.zeros(7, np.int64)
    count_set(lib, c, [fan(13, 12, 20, 1)], 5)
    ok(lib.acc_motif_last_stats(c.h, P(stats)), "last_stats")
    c.close()
    return int(stats[2])


def host_k5_sparse(lib):
    """How often the list scan counted a uniform graph of 90 arcs on 80 vertices, and
    one of 400 arcs (k = 5)."""
    from tests.emu.lib_scenarios import Ctx
    rng = np.random.default_rng(8)
    scans = []
    for m in (90, 400):
        key = rng.permutation(80 * 79)[:m]
        s, d = key // 79, key % 79
        c = Ctx(lib)
        count_set(lib, c, [(80, s, d + (d >= s))], 5)
        c.close()
        scans.append(lib.emu_scan_count())
    return scans


def host_k5_scanned(lib):
    """Neighbour entries read for a k = 5 graph: on its own, and by the list scan
    of a set with a second, empty graph; how often a scan followed the passes."""
    from tests.emu.lib_scenarios import Ctx, P, ok
    c = Ctx(lib)
    stats = np.zeros(7, np.int64)
    read = []
    for gs in ([fan(13, 12, 20, 1)], [fan(13, 12, 20, 1), (1, np.zeros(0, np.int64), np.zeros(0, np.int64))]):
        count_set(lib, c, gs, 5)
        ok(lib.acc_motif_last_stats(c.h, P(stats)), "last_stats")
        read.append(int(stats[6]))
    c.close()
    return read + [lib.emu_scan_count()]


def host_autotune(lib):
    """The schedule before and after the autotuner, and what it returned, by what
    counts the batch."""
    import paper_1203_3415_gb300 as acc
    from tests.emu.lib_scenarios import Ctx, _descs, ok
    c = Ctx(lib)
    seen = []
    g = fan(6, 4, 8, 1)
    for mode, k, gs in ((acc.ACC_MODE_COUNT, 4, [g, g]), (acc.ACC_MODE_COUNT, 5, [g]), (acc.ACC_MODE_FORMULA, 3, [g, g]),
                        (acc.ACC_MODE_ENUMERATE, 3, [g, g])):
        light, target, ms = ctypes.c_int64(), ctypes.c_int64(), ctypes.c_float()
        ok(lib.acc_ctx_set_mode(c.h, mode), "set_mode")
        ok(lib.acc_ctx_set_schedule(c.h, 777, 999), "set_schedule")
        descs, keep = _descs(gs)
        ok(lib.acc_motif_batch_prepare(c.h, descs, len(gs), k, None), "batch_prepare")
        ok(lib.acc_motif_batch_autotune(c.h, None, ctypes.byref(light), ctypes.byref(target), ctypes.byref(ms)), "autotune")
        pair = [light.value, target.value]
        ok(lib.acc_ctx_get_schedule(c.h, ctypes.byref(light), ctypes.byref(target)), "get_schedule")
        assert pair == [light.value, target.value] and ms.value > 0.0
        seen.append(pair)
    c.close()
    return seen


def host_short_memory(lib):
    """Counts of sets that fit the device's memory until their pattern counters are
    added: bytes held where there is no limit, and the least limit under which the
    counts are right (below it the call says so)."""
    import paper_1203_3415_gb300 as acc
    from tests.emu.lib_scenarios import Ctx, NCLS, P, _descs
    lib.emu_bytes.restype = ctypes.c_ulonglong
    lib.emu_limit.argtypes = [ctypes.c_ulonglong]
    out = []
    for k, gs, steps in ((4, [fan(40, 20, 30, 2)] * 2, 10), (5, [fan(8, 6, 10, 1)], 4)):
        table = Ctx(lib)  # (the class tables stay)
        for kk in (3, 4, 5):
            assert lib.acc_motif_prepare(table.h, kk, None) == 0
        before = lib.emu_bytes()
        want = [oracle.count(*g, k) for g in gs]
        descs, keep = _descs(gs)
        counts, st = np.zeros((len(gs), NCLS[k]), np.int64), np.full(1, -1, np.int32)

        def count(limit):
            lib.emu_limit(limit)
            c = Ctx(lib)
            rc = lib.acc_motif_count_batch(c.h, descs, len(gs), k, None, P(counts), P(st))
            if rc == 0:
                assert st[0] == 0 and all(np.array_equal(o, w) for o, w in zip(counts, want)), limit
            held = lib.emu_bytes() - before
            c.close()
            lib.emu_limit(1 << 63)
            assert rc in (0, acc.ACC_ERR_NOMEM), rc
            return rc == 0, held
        held = count(1 << 63)[1]
        limit = held
        while count(before + limit - held // steps)[0]:
            limit -= held // steps
        out.append([held, limit])
        table.close()
    return out


def host_footprint(lib):
    """Bytes held by a slot's context after it was made ready for a sequence of
    (n, m, k), over its footprint before the last; the most of all sequences."""
    from tests.emu.lib_scenarios import Ctx, ok
    lib.emu_bytes.restype = lib.emu_footprint.restype = ctypes.c_longlong
    lib.emu_reserve.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    lib.emu_footprint.argtypes = lib.emu_reserve.argtypes + [ctypes.c_int]
    tables = Ctx(lib)
    ok(lib.acc_motif_prepare(tables.h, 5, None), "prepare")
    most = 0.0
    for graphs in ([(3000, 400000)], [(3000, 9000)], [(20000, 300000)], [(19000, 90000), (2000, 500000)]):
        for ks in ((3, 4, 5), (5, 4, 3), (4, 5), (5,), (4,)):
            for ways in range(3):  # (scan, as ruled, either)
                for at_once in (False, True):
                    c = Ctx(lib)
                    before = lib.emu_bytes()
                    for n, m in graphs:
                        fp = lib.emu_footprint(c.h, n, m, min(ks), max(ks), ways)
                        for k in ks:
                            if not at_once:
                                fp = lib.emu_footprint(c.h, n, m, k, k, ways)
                            ok(lib.emu_reserve(c.h, n, m, k, ways), "reserve")
                            most = max(most, (lib.emu_bytes() - before) / (fp + 4096.0))
                    c.close()
    tables.close()
    return most


def host_dense_block(lib):
    """Whether the workspace of a graph of 20000 vertices and m arcs has the dense
    block."""
    from tests.emu.lib_scenarios import Ctx, ok
    lib.emu_bytes.restype = ctypes.c_longlong
    lib.emu_reserve.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    tables = Ctx(lib)
    ok(lib.acc_motif_prepare(tables.h, 5, None), "prepare")
    seen = []
    for k, m in ((3, 400000), (3, 400001), (4, 200000), (4, 200001)):
        c = Ctx(lib)
        before = lib.emu_bytes()
        ok(lib.emu_reserve(c.h, 20000, m, k, 1), "reserve")
        seen.append(lib.emu_bytes() - before > 20000 ** 2 // 4)
        c.close()
    # no memory for the block: the sparse build after all
    lib.emu_limit.argtypes = [ctypes.c_ulonglong]
    c = Ctx(lib)
    before = lib.emu_bytes()
    lib.emu_limit(before + 20000 ** 2 // 4)
    ok(lib.emu_reserve(c.h, 20000, 200001, 4, 1), "reserve")
    lib.emu_limit(1 << 63)
    seen.append(lib.emu_bytes() - before > 20000 ** 2 // 4)
    c.close()
    tables.close()
    return seen


def host_server_budget(lib):
    """A server whose budget holds the list scan's workspace, not the pattern
    counters: the request's state, and whether patterns counted it."""
    from tests.emu.lib_scenarios import Ctx, P, csr, ok
    n = 1024
    key = np.random.default_rng(3).permutation(n * (n - 1))[:8000]
    src, dst = key // (n - 1), key % (n - 1)
    dst = dst + (dst >= src)
    rp, cl = csr(n, src, dst)
    lib.emu_footprint.restype = ctypes.c_longlong
    lib.emu_footprint.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_int,
                                  ctypes.c_int]
    c = Ctx(lib)
    scan, patterns = (lib.emu_footprint(c.h, n, len(cl), 4, 4, ways) for ways in (0, 1))
    c.close()
    seen = []
    for budget in (scan, patterns):
        srv, gid, rid, state = ctypes.c_void_p(), ctypes.c_int32(), ctypes.c_int64(), ctypes.c_int32()
        out = np.zeros(199, np.int64)
        before = lib.emu_partial_count()
        ok(lib.acc_server_create(ctypes.byref(srv), 0, 1, budget), "server_create")
        ok(lib.acc_server_add_graph(srv, P(rp), P(cl), n, len(cl), ctypes.byref(gid)), "add_graph")
        ok(lib.acc_server_submit(srv, gid.value, 4, ctypes.byref(rid)), "submit")
        ok(lib.acc_server_drain(srv), "drain")
        ok(lib.acc_server_poll(srv, rid, ctypes.byref(state), P(out), None), "poll")
        lib.acc_server_destroy(srv)
        assert state.value < 0 or np.array_equal(out, oracle.count(n, src, dst, 4))
        seen.append([state.value, lib.emu_partial_count() > before])
    return [scan < patterns] + seen


def host_reserved(lib):
    """Bytes a server grows by when it serves, after the reserve, a k = 5 request on
    the smaller of two graphs, which has more arcs a vertex; whether it was scanned."""
    from tests.emu.lib_scenarios import P, csr, ok
    lib.emu_bytes.restype = ctypes.c_longlong
    rng = np.random.default_rng(3)
    srv, gid, rid, state = ctypes.c_void_p(), ctypes.c_int32(), ctypes.c_int64(), ctypes.c_int32()
    ok(lib.acc_server_create(ctypes.byref(srv), 0, 1, 1 << 30), "server_create")
    graphs = []
    for n, m in ((3000, 2600), (1024, 2500)):
        key = rng.permutation(n * (n - 1))[:m]
        src, dst = key // (n - 1), key % (n - 1)
        graphs.append((n, src, dst + (dst >= src)))
        arrays = csr(*graphs[-1])
        graphs.append(arrays)
        ok(lib.acc_server_add_graph(srv, P(arrays[0]), P(arrays[1]), n, m, ctypes.byref(gid)), "add_graph")
    ok(lib.acc_server_reserve(srv), "reserve")
    before = lib.emu_bytes()
    ok(lib.acc_server_submit(srv, gid.value, 5, ctypes.byref(rid)), "submit")
    ok(lib.acc_server_drain(srv), "drain")
    more = lib.emu_bytes() - before
    out = np.zeros(9364, np.int64)
    ok(lib.acc_server_poll(srv, rid, ctypes.byref(state), P(out), None), "poll")
    lib.acc_server_destroy(srv)
    assert np.array_equal(out, oracle.count(*graphs[2], 5))
    return [more, lib.emu_scan_count()]


def host_own_stream(lib):
    """Batches and randomised copies on a stream that does not wait for the legacy
    one; edges of the last batch's graphs, as the statistics have them."""
    import paper_1203_3415_gb300 as acc
    from tests.emu.lib_scenarios import Ctx, NCLS, P, _descs, csr, ok
    lib.emu_stream_create.restype = ctypes.c_void_p
    s = ctypes.c_void_p(lib.emu_stream_create())
    c = Ctx(lib)
    for gs in ([fan(6, 4, 8, 1), fan(5, 3, 9, 2)], [fan(4, 4, 7, 3), fan(7, 2, 8, 4), fan(3, 3, 3, 5)]):
        descs, keep = _descs(gs)
        counts = np.full((len(gs), NCLS[4]), -1, np.int64)
        ok(lib.acc_motif_batch_prepare(c.h, descs, len(gs), 4, s), "batch_prepare")
        ok(lib.acc_motif_batch_run(c.h, s, P(counts), None), "batch_run")
        for o, g in zip(counts, gs):
            assert np.array_equal(o, oracle.count(*g, 4))
        arrays = [csr(*g) for g in gs]
        R, seeds, m = 2, np.arange(len(gs), dtype=np.uint64), sum(len(a[1]) for a in arrays)
        out, accepted = np.zeros(R * m, np.int32), np.zeros(len(gs) * R, np.int64)
        ok(lib.acc_swap_randomise(c.h, descs, len(gs), R, 2, P(seeds), acc.ACC_RAND_SWAP, s, P(out), P(accepted), None),
           "swap_randomise")
        want = [oracle.swap_randomise(g[0], *a, 2 * len(a[1]), i + r)[0] for i, (g, a) in enumerate(zip(gs, arrays))
                for r in range(R)]
        assert np.array_equal(out, np.concatenate(want))
    stats = np.zeros(7, np.int64)
    ok(lib.acc_motif_last_stats(c.h, P(stats)), "last_stats")
    c.close()
    pairs = [np.unique(np.minimum(g[1], g[2]) * g[0] + np.maximum(g[1], g[2])) for g in gs]
    return [int(stats[3]), sum(len(p) for p in pairs)]


def host_two_devices(lib):
    """The same counts on device 0, then on device 1: kernels whose limit of shared
    memory was raised on the first, and on both."""
    from tests.emu.lib_scenarios import Ctx, ok

    class On(Ctx):
        def __init__(self, lib, device):
            self.lib, self.h = lib, ctypes.c_void_p()
            ok(lib.acc_ctx_create(ctypes.byref(self.h), device), "acc_ctx_create")
    g, big = fan(6, 4, 8, 1), fan(13, 12, 1200, 1)
    for device in (0, 1):
        c = On(lib, device)
        count_set(lib, c, [big, big], 3)
        count_set(lib, c, [g, g], 4)
        count_set(lib, c, [g], 4)
        count_set(lib, c, [g], 5)
        c.close()
    first, both = ctypes.c_int(), ctypes.c_int()
    lib.emu_limit_counts(ctypes.byref(first), ctypes.byref(both))
    return [first.value, both.value]


def host_many_graphs(lib):
    """Sets of `graphs` graphs of n vertices and m arcs: counted by partial patterns?"""
    from tests.emu.lib_scenarios import Ctx
    rng = np.random.default_rng(5)
    c = Ctx(lib)
    seen = []
    for k, graphs, n, m in SETS:
        gs = []
        for _ in range(graphs):
            key = rng.permutation(n * (n - 1))[:m]
            s, d = key // (n - 1), key % (n - 1)
            gs.append((n, s, d + (d >= s)))
        before = lib.emu_partial_count()
        count_set(lib, c, gs, k)
        seen.append(lib.emu_partial_count() > before)
    c.close()
    return seen


# --------------------------------------------------------------------------
# tests
# --------------------------------------------------------------------------

# (EMU_SCHED 0: the threads of a block arrive in ascending order, so warps 0 and 1
# have passed when thread 64 does; 1: in descending order, all but warp 0)
RAISED = [(phase, order, at) for phase in (1, 2) for order, at in ((0, 64), (1, 31))]
for phase, order, at in RAISED:
    RUNS["raised", phase, order, at] = ("k5_scans", dict(EMU_SCHED=order, EMU_RAISE_PHASE=phase, EMU_RAISE_AT=at))
RUNS["not raised"] = ("k5_scans", {})


@pytest.mark.parametrize("phase,order,at", RAISED)
def test_return_to_the_scan_raised_as_a_block_starts(on_host, phase, order, at):
    """The 5-cycle pass while another block or kernel raises the return to the
    list scan: each block goes on or leaves as a whole."""
    assert on_host(("raised", phase, order, at)) == 1


def test_no_return_to_the_scan(on_host):
    assert on_host("not raised") == 0


RUNS["rows"] = ("k5_scanned", dict(EMU_ROWS=8))


def test_graphs_with_large_hubs_pay_for_the_scan_alone(on_host):
    """k = 5, a root of more rows than the 5-cycle tables count: the passes leave at
    once, and what is read is what the list scan reads."""
    alone, scan, returned = on_host("rows")
    assert returned == 1 and alone == scan > 0


RUNS["autotune"] = ("autotune", {})


def test_autotuner_keeps_the_schedule_that_no_scan_reads(on_host):
    *unread, scanned = on_host("autotune")
    assert unread == [[777, 999]] * 3 and scanned != [777, 999]


RUNS["memory"] = ("short_memory", {})


def test_sets_whose_counters_do_not_fit_are_scanned(on_host):
    for held, least in on_host("memory"):
        assert least < 0.8 * held


# (one emulated SM: k = 4 from 5 graphs on, k = 3 from 17)
SETS = [(4, 5, 32, 63), (4, 5, 32, 64), (4, 5, 31, 95), (4, 5, 31, 96), (4, 4, 10, 20), (3, 17, 12, 47), (3, 17, 12, 48),
        (3, 16, 12, 20)]
RUNS["many"] = ("many_graphs", {})


def test_sets_of_many_tiny_graphs_are_scanned(on_host):
    assert on_host("many") == [False, True, False, True, True, False, True, True]


RUNS["sparse"] = ("k5_sparse", {})


def test_sparse_uniform_graphs_are_scanned(on_host):
    """k = 5, sum of d (d - 1) (d - 2) / 2 below 15 a vertex: left to the scan."""
    assert on_host("sparse") == [1, 1]


RUNS["devices"] = ("two_devices", {})


def test_every_device_gets_the_kernels_shared_memory(on_host):
    first, both = on_host("devices")
    assert first == both > 20


RUNS["footprint"] = ("footprint", {})
RUNS["budget"] = ("server_budget", {})


def test_footprint_covers_what_a_slot_holds(on_host):
    assert on_host("footprint") <= 1.0


def test_requests_that_fit_by_the_scan_alone_are_served(on_host):
    import paper_1203_3415_gb300 as acc
    done = acc.ACC_REQ_DONE
    assert on_host("budget") == [True, [done, False], [done, True]]


RUNS["reserved"] = ("reserved", dict(EMU_ARCS1=10000))


def test_serving_allocates_nothing_after_the_reserve(on_host):
    """k = 5, a registered graph that is counted by partial patterns where the
    largest of both sizes would not be."""
    assert on_host("reserved") == [0, 0]


RUNS["stream"] = ("own_stream", dict(EMU_DEFER=1))


def test_host_tables_are_copied_on_the_stream_that_reads_them(on_host):
    seen, edges = on_host("stream")
    assert seen == edges


RUNS["parts"] = ("k5_parts", {})


def test_statistics_have_the_parts_of_every_pass(on_host):
    assert on_host("parts") >= 1


RUNS["returns", 0] = ("returns", {})
RUNS["returns", 1] = ("returns", dict(EMU_TRIANGLES=5))
RUNS["returns", 2] = ("returns", dict(EMU_RANGES=1))
RUNS["wide"] = ("wide", dict(EMU_FIELD=20))


@pytest.mark.parametrize("limit,scans", [(0, [0, 0]), (1, [1, 0]), (2, [0, 1])], ids=["none", "triangles", "ranges"])
def test_full_lists_return_to_the_scan(on_host, limit, scans):
    assert on_host(("returns", limit)) == scans


def test_sets_with_wide_roots(on_host):
    assert on_host("wide") == 0


@pytest.mark.gpu
def test_set_with_a_root_of_1100_rows():
    """k = 3, 4, a set of graphs, one with a root of more rows than a table's 10-bit
    fields count, against the enumerate mode."""
    import torch
    from paper_1203_3415_gb300 import build
    build.build()
    import paper_1203_3415_gb300 as acc
    import synth
    gs = [fan(1100, 3, 900, 1), fan(300, 6, 500, 2)]
    small = synth.chung_lu(500, 2000, 2.2, 60, 10, 5)
    gs.append((small.n, small.src, small.dst))
    from tests.emu.lib_scenarios import csr
    dev = [(torch.from_numpy(r).cuda(), torch.from_numpy(c).cuda(), g[0]) for g in gs for r, c in [csr(*g)]]
    c = acc.Counter(0)
    try:
        for k in (3, 4):
            got = {}
            for mode in (acc.ACC_MODE_COUNT, acc.ACC_MODE_ENUMERATE):
                c.set_mode(mode)
                c.prepare_batch(dev, k)
                got[mode] = c.run_batch().cpu().numpy().tolist()
            assert got[acc.ACC_MODE_COUNT] == got[acc.ACC_MODE_ENUMERATE], k
    finally:
        c.close()


RUNS["dense"] = ("dense_block", {})


def test_sparse_build_up_to_its_arcs_a_vertex(on_host):
    """(from 20000 vertices here)"""
    assert on_host("dense") == [False, True, False, True, False]


if __name__ == "__main__":
    import paper_1203_3415_gb300 as acc
    lib = acc.declare(ctypes.CDLL(sys.argv[1]))
    print("\n" + json.dumps(globals()["host_" + sys.argv[2]](lib)))
