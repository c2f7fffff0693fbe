"""The counts by partial patterns (csrc/partial.cu, csrc/partial5.cu), exact
integers throughout, on graphs at the edges of its tables: roots with as many wedges
as a warp's or a block's table takes and one more, roots cut into ranges of
end vertices, roots with more rows than a table's 10-bit fields count, ends
shared by all rows of a root, and queues too short for every part.

On the CPU the library's own source runs on the host (tests/emu) with the
size threshold at 0, against the oracle; on the GPU against the enumerate
mode, which visits every subset."""
import ctypes
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import oracle
import synth
from tests.graph_helpers import complete_bidirected, random_digraph

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def fan(rows, ends, pool, seed, filler=0):
    """Vertex 0 with `rows` neighbours that have `ends` further neighbours each
    out of `pool` vertices, random states; plus a random digraph of `filler`
    vertices and 3 arcs each."""
    rng = np.random.default_rng(seed)
    s, d = [], []

    def edge(a, b):
        r = int(rng.integers(0, 3))
        if r != 1:
            s.append(a), d.append(b)
        if r != 0:
            s.append(b), d.append(a)

    for i in range(rows):
        edge(0, 1 + i)
        for e in rng.permutation(pool)[:ends]:
            edge(1 + i, 1 + rows + int(e))
    n = 1 + rows + pool
    if filler:
        a, b = rng.integers(0, filler, 3 * filler), rng.integers(0, filler, 3 * filler)
        s.extend((n + a[a != b]).tolist()), d.extend((n + b[a != b]).tolist())
        n += filler
    return n, np.asarray(s, np.int64), np.asarray(d, np.int64)


def small_sets(k):
    rng = np.random.default_rng(70 + k)
    gs = []
    if k == 5:  # (the host runs about 10^5 device threads a graph: few and small ones)
        s, d = random_digraph(rng, 14, p=0.4, recip=0.5)
        gs.append((14, np.asarray(s, np.int64), np.asarray(d, np.int64)))
        g = synth.chung_lu(150, 500, 2.1, 60, 20, 4)
        return gs + [(g.n, g.src, g.dst), fan(13, 12, 20, 1)]
    for _ in range(7):
        n = int(rng.integers(2, 32))
        s, d = random_digraph(rng, n, p=float(rng.uniform(0.02, 0.6)), recip=float(rng.random()))
        gs.append((n, np.asarray(s, np.int64), np.asarray(d, np.int64)))
    gs.insert(3, (5, np.zeros(0, np.int64), np.zeros(0, np.int64)))
    gs.append(fan(13, 12, 20, 1))   # 156 wedges: more than a warp's table
    gs.append(fan(40, 20, 30, 2))   # 800: more than a block's, and few ends
    gs.append(fan(60, 30, 900, 3))  # ranges of ends
    g = synth.chung_lu(150, 600, 2.1, 60, 20, 4)
    gs.append((g.n, g.src, g.dst))
    s, d = complete_bidirected(24)
    gs.append((24, np.asarray(s), np.asarray(d)))
    return gs


@pytest.fixture(scope="module", params=["-DACC_CYCLE_SLOTS=256", "-DACC_QUEUE_CAP=3ull"],
                ids=["short_tables", "short_queue"])
def host_lib(request, tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    from tests.test_cpu_emulation import CSRC, EMU, _launches_to_calls
    out = tmp_path_factory.mktemp("partial")
    units = [os.path.join(EMU, "emu_rt.cpp")]
    for name in sorted(os.listdir(CSRC)):
        if name.endswith(".cu"):
            units.append(str(out / (name[:-3] + ".cpp")))
            open(units[-1], "w").write('#include "shim.h"\n' + _launches_to_calls(open(os.path.join(CSRC, name)).read()))
    asan = subprocess.run(["g++", "-print-file-name=libasan.so"], capture_output=True, text=True).stdout.strip()
    san = ["-fsanitize=address", "-DEMU_EXACT_ALLOC", "-DEMU_LANE_STACK=65536"] if os.path.isabs(asan) else []
    procs = [subprocess.Popen(["g++", "-std=c++20", "-O1", "-fPIC", "-pthread", "-w", *san, "-DACC_PARTIAL_MIN_ARCS=0",
                               request.param, "-I", EMU, "-I", os.path.join(EMU, "fake"), "-I", CSRC, "-c", u,
                               "-o", str(out / f"u{i}.o")], stderr=subprocess.PIPE, text=True) for i, u in enumerate(units)]
    for p in procs:
        err = p.communicate()[1]
        assert p.returncode == 0, err[-3000:]
    so = str(out / "lib.so")
    subprocess.run(["g++", "-shared", "-pthread", *san[:1], "-o", so] +
                   [str(out / f"u{i}.o") for i in range(len(units))], check=True)
    return so, dict(os.environ, PYTHONPATH=ROOT, **({"LD_PRELOAD": asan, "ASAN_OPTIONS": "detect_leaks=0"} if san else {}))


@pytest.mark.parametrize("k", [3, 4, 5])
def test_partial_patterns_on_the_host(host_lib, k):
    so, env = host_lib
    r = subprocess.run([sys.executable, os.path.abspath(__file__), so, str(k)], cwd=ROOT, env=env, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, (r.stdout + r.stderr)[-3000:]


def host_main(so, k):
    import paper_1203_3415_gb300 as acc
    from tests.emu.lib_scenarios import NCLS, P, Ctx, _descs, ok, sync
    lib = acc.declare(ctypes.CDLL(so))
    gs = small_sets(k)
    want = [oracle.count(n, s, d, k) for n, s, d in gs]
    for adj in (acc.ACC_ADJ_AUTO, acc.ACC_ADJ_HASH, acc.ACC_ADJ_SPARSE)[k == 5:]:
        c = Ctx(lib)
        ok(lib.acc_ctx_set_adjacency(c.h, adj), "set_adjacency")
        # (a set of several graphs for k = 3, 4, one graph at a time for k = 5)
        for sets in ([list(range(len(gs)))] if k < 5 else [[i] for i in range(len(gs))]):
            descs, keep = _descs([gs[i] for i in sets])
            ok(lib.acc_motif_batch_prepare(c.h, descs, len(sets), k, None), "batch_prepare")
            for rep in range(2 if k < 5 else 1):
                out, st = np.zeros((len(sets), NCLS[k]), np.int64), np.full(1, -1, np.int32)
                ok(lib.acc_motif_batch_run(c.h, None, P(out), P(st)), "batch_run")
                sync(lib)
                assert st[0] == 0
                for o, i in zip(out, sets):
                    assert np.array_equal(o, want[i]), (adj, rep, i)
        c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("rows,ends,pool", [(12, 12, 400), (29, 5, 400), (31, 22, 500), (683, 1, 400), (200, 20, 2500),
                                            (400, 40, 60), (1023, 3, 900), (1024, 3, 900), (1100, 2, 2), (1500, 7, 3000)])
def test_partial_patterns_equal_the_walk(rows, ends, pool):
    from paper_1203_3415_gb300 import build
    build.build()
    import paper_1203_3415_gb300 as acc
    from tests.gpu_helpers import gpu_count
    n, s, d = fan(rows, ends, pool, rows + ends, filler=6000)
    c = acc.Counter(0)
    try:
        # (k = 5: not where the walk would visit 10^12 subsets; 1024 rows go to the scan)
        for k in (3, 4, 5) if rows * ends < 10000 and pool > 60 else (3, 4):
            c.set_mode(acc.ACC_MODE_ENUMERATE)
            c.set_adjacency(acc.ACC_ADJ_AUTO)
            want = gpu_count(c, n, s, d, k).tolist()
            c.set_mode(acc.ACC_MODE_COUNT)
            for adj in (acc.ACC_ADJ_AUTO, acc.ACC_ADJ_HASH, acc.ACC_ADJ_SPARSE):
                c.set_adjacency(adj)
                assert gpu_count(c, n, s, d, k).tolist() == want, (k, adj)
    finally:
        c.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [98303, 98304])
def test_sparse_build_from_98304_vertices(n):
    """k = 3, 4 on either side of the size from which partial patterns are
    counted on sorted rows: the dense block's counts, also when repeated (the
    count is replayed) and after another graph."""
    import torch
    from paper_1203_3415_gb300 import build
    build.build()
    import paper_1203_3415_gb300 as acc
    g = synth.chung_lu(n, 2 * n, 2.2, 300, 10, 31)
    rowptr, col = g.csr()
    r, cl = torch.from_numpy(rowptr).cuda(), torch.from_numpy(col).cuda()
    a, dense = acc.Counter(0), acc.Counter(0)
    dense.set_adjacency(acc.ACC_ADJ_DENSE)
    try:
        for k in (3, 4):
            want = dense.count(r, cl, g.n, k).cpu().numpy().tolist()
            out = torch.zeros(acc.NUM_CLASSES[k], dtype=torch.int64, device="cuda")
            for _ in range(4):
                out.zero_()
                assert a.count(r, cl, g.n, k, counts=out).cpu().numpy().tolist() == want
    finally:
        a.close()
        dense.close()


if __name__ == "__main__":
    host_main(sys.argv[1], int(sys.argv[2]))
