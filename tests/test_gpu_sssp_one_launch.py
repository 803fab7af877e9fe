"""db_sssp of hypersparse handles in one launch: rows and columns longer than a listed chunk, without the row-run
index (push steps only), unit weights, and the same steps as the host loop of (min, +) products makes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, ref_matrix

pytestmark = pytest.mark.gpu


def star_and_noise(n, seed):
    """Vertex 5 touches every other vertex in both directions; sparse random edges beside it."""
    bg = wl.random_sparse(n, n, 3 * n, seed)
    rows = np.r_[bg.rows(), np.full(n - 1, 5), np.delete(np.arange(n), 5)]
    cols = np.r_[bg.col_idx, np.delete(np.arange(n), 5), np.full(n - 1, 5)]
    keys = wl.sorted_unique(rows.astype(np.int64) * n + cols)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    return wl.CSR(n, n, ptr, idx, (1 + (wl.rand_u64(seed, 3, np.arange(keys.size)) % 63)).astype(np.float32) / 8.0)


@pytest.mark.parametrize("n", [1031, 40001])
@pytest.mark.parametrize("dtype", [B.F32, B.PATTERN])
@pytest.mark.parametrize("no_index", [0, 1])
def test_sssp_one_launch(n, dtype, no_index):
    csr = star_and_noise(n, 4)
    if dtype == B.PATTERN:
        csr.val = np.ones(csr.nnz, np.float32)
    o = B.default_create_opts()
    o.no_bfs_index = no_index
    h = Handle(csr, dtype, opts=o)
    A = ref_matrix(csr)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    for src in (5, 0, n - 1):
        steps = []
        for path in (B.PATH_AUTO, B.PATH_PUSH):
            h.set_opts(force_path=path)
            steps.append(B.db_sssp(h.h, src, dist))
            torch.cuda.synchronize()
            assert np.array_equal(dist.cpu().numpy().astype(np.float64), oracle.ref_sssp(A, src))
        assert steps[0] == steps[1]
    h.close()


@pytest.mark.parametrize("low", [-np.inf, -3.4e38, np.inf])
def test_rows_that_begin_with_extreme_weights(low):
    """Rows of a pulled step whose first elements, of the lowest (or highest) weights there are, lead to vertices that were never
    reached: the search goes on to the finite ones behind them."""
    n = 4000
    rng = np.random.default_rng(2)
    mid = np.arange(1, 1501)
    rows = [mid, rng.integers(1501, 3000, 4 * mid.size), np.repeat(np.arange(1501, 1601), 12), [3500]]
    cols = [np.zeros(mid.size, np.int64), np.repeat(mid, 4), np.tile(np.arange(3001, 3013), 100), [1550]]
    kind = np.r_[np.zeros(mid.size), np.zeros(4 * mid.size), np.ones(1200), [0]]
    key = np.concatenate(rows).astype(np.int64) * n + np.concatenate(cols)
    keys, at = np.unique(key, return_index=True)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    val = np.where(kind[at] == 1, low, (1 + rng.integers(0, 63, keys.size)) / 8.0).astype(np.float32)
    h = Handle(wl.CSR(n, n, ptr, idx, val), B.F32)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    want = np.full(n, np.inf, np.float32)
    want[0] = 0.0
    r = np.repeat(np.arange(n), np.diff(ptr))
    for _ in range(4):                                       # (no path has more than three edges)
        new = want.copy()
        live = np.isfinite(want[idx])
        np.minimum.at(new, r[live], want[idx[live]] + val[live])
        want = new
    for path in (B.PATH_AUTO, B.PATH_PUSH):
        h.set_opts(force_path=path)
        B.db_sssp(h.h, 0, dist)
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy(), want)
    assert np.isfinite(want[1501:1601]).sum() > 90
    h.close()


@pytest.mark.parametrize("fan", [1, 1023, 1024, 1025, 6000])
@pytest.mark.parametrize("dtype", [B.F32, B.PATTERN])
def test_listed_and_unlisted_frontiers(fan, dtype):
    """Frontiers at the length up to which a step's marked vertices are kept as a list, in turn with longer and shorter ones: the source
    reaches `fan` vertices, they reach a third of that and one vertex with a long column, then single vertices; a part that is not reached keeps the
    pushed steps a small share of the elements.  (Dyadic weights: every path sum is exact.)"""
    n = 40011
    rng = np.random.default_rng(fan)
    a = 16 + np.arange(fan)
    b = 8000 + np.arange(max(1, fan // 3))
    u = [np.full(fan, 3), a, np.full(1, a[0]), np.full(700, 20000), [20001, 20002, 20003], rng.integers(22000, n, 300000)]
    v = [a, b[rng.integers(0, b.size, fan)], [20000], 20001 + np.arange(700), [21000, 21001, 21002], rng.integers(22000, n, 300000)]
    keys = wl.sorted_unique(np.concatenate(v).astype(np.int64) * n + np.concatenate(u))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    val = np.ones(keys.size, np.float32) if dtype == B.PATTERN else (1 + rng.integers(0, 63, keys.size)).astype(np.float32) / 8.0
    csr = wl.CSR(n, n, ptr, idx, val)
    h, A = Handle(csr, dtype), ref_matrix(csr)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    for src in (3, 20000, int(a[-1])):
        steps = []
        for path in (B.PATH_AUTO, B.PATH_PUSH, B.PATH_AUTO):
            h.set_opts(force_path=path)
            steps.append(B.db_sssp(h.h, src, dist))
            torch.cuda.synchronize()
            assert np.array_equal(dist.cpu().numpy().astype(np.float64), oracle.ref_sssp(A, src))
        assert steps[0] == steps[1] == steps[2]
    h.close()


@pytest.mark.parametrize("length", [1, 3, 4, 31, 32, 33, 63, 64, 65, 543, 545, 1100, 2600])
def test_rows_of_a_pulled_step(length):
    """Rows at the lengths where a lane hands a row over and where what is left of it is one chunk or several, dense blocks among their elements; the
    vertices they lie behind are reached in one step, so that the next one is pulled, and once more with better distances a step later."""
    rows_of_a_pulled_step(6007, length)


@pytest.mark.parametrize("length", [3, 16, 17, 29, 33, 65, 129, 545])
@pytest.mark.parametrize("lanes", [8, 4, 2, 1, 0])
def test_lanes_that_share_a_row_of_a_pulled_step(length, lanes):
    """The same rows in graphs of as many vertices as leave two, four or eight lanes of the GPU for each, with the last rows at the end of the range, and of one more than it has lanes."""
    threads = 1024 * torch.cuda.get_device_properties(0).multi_processor_count
    rows_of_a_pulled_step(threads // lanes if lanes else threads + 1, length)


def rows_of_a_pulled_step(n, length):
    rng = np.random.default_rng(length)
    src, late = 0, 1
    mid = np.arange(32, 32 + 2700)                         # reached from the source; half of them again, for less, by way of `late`
    rows = [mid, [late], mid[::2], np.repeat(np.arange(3000, 3200), length), np.repeat(np.arange(3200, 3232), 32)]
    cols = [np.zeros(mid.size), [src], np.full(mid[::2].size, late), np.concatenate([rng.choice(mid, length, replace=False) for _ in range(200)]),
            np.tile(np.arange(32, 64), 32)]
    key = np.concatenate(rows).astype(np.int64) * n + np.concatenate(cols).astype(np.int64)
    keys = wl.sorted_unique(key)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    val = (8 + rng.integers(0, 500, keys.size)).astype(np.float32) / 8.0
    r = np.repeat(np.arange(n), np.diff(ptr))
    val[(r == late) | (idx == late)] = 1.0 / 8.0
    csr = wl.CSR(n, n, ptr, idx, val)
    h, A = Handle(csr, B.F32), ref_matrix(csr)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    steps = []
    for path in (B.PATH_AUTO, B.PATH_PUSH):
        h.set_opts(force_path=path)
        steps.append(B.db_sssp(h.h, src, dist))
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy().astype(np.float64), oracle.ref_sssp(A, src))
    assert steps[0] == steps[1]
    h.close()


@pytest.mark.parametrize("length", [40, 333, 1200])
@pytest.mark.parametrize("base", [4096.0, -4096.0])
def test_many_pulled_steps_in_a_row(length, base):
    """A path whose vertices also have an edge each from the source, of weights that rise twice as fast as the path's: every step improves all that is left of it, so the
    steps are pulled one after the other -- 1200 of them in more than one launch -- until the frontier is a few vertices, the path's end and a tail behind it.
    (Distances of both signs; whole numbers: every sum is exact.)"""
    n = length + 107
    k = np.arange(length)
    rows = np.r_[1 + k, 2 + k[:-1], length + 1 + np.arange(6)]
    cols = np.r_[np.zeros(length, np.int64), 1 + k[:-1], length + np.arange(6)]
    val = np.r_[base + 2.0 * k, np.ones(length - 1), np.full(6, 3.0)].astype(np.float32)
    order = np.argsort(rows.astype(np.int64) * n + cols)
    ptr, idx = wl.csr_from_sorted_keys(n, n, (rows.astype(np.int64) * n + cols)[order])
    want = np.full(n, np.inf, np.float32)
    want[0] = 0.0
    want[1:length + 1] = base + k
    want[length + 1:length + 7] = base + length - 1 + 3.0 * (1 + np.arange(6))
    h = Handle(wl.CSR(n, n, ptr, idx, val[order]), B.F32)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    steps = []
    for path in (B.PATH_AUTO, B.PATH_PUSH, B.PATH_AUTO):
        h.set_opts(force_path=path)
        steps.append(B.db_sssp(h.h, 0, dist))
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy(), want)
    assert steps[0] == steps[1] == steps[2] and steps[0] > length
    h.close()


def check_steps(csr, src, repeats=1):
    """Distances and steps of the one launch against the oracle and the host loop's."""
    h, A = Handle(csr, B.F32), ref_matrix(csr)
    want = oracle.ref_sssp(A, src)
    dist = torch.empty(csr.n, dtype=torch.float32, device="cuda")
    steps = []
    for path in [B.PATH_PUSH] + [B.PATH_AUTO] * repeats:
        h.set_opts(force_path=path)
        steps.append(B.db_sssp(h.h, src, dist))
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy().astype(np.float64), want)
    assert len(set(steps)) == 1
    h.close()


def graph(n, edges):
    """CSR of {(from, to): weight}, an edge each."""
    u, v, w = (np.concatenate([np.broadcast_to(e[i], np.broadcast_shapes(*(np.shape(q) for q in e))).ravel() for e in edges]) for i in range(3))
    keys, at = np.unique(v.astype(np.int64) * n + u.astype(np.int64), return_index=True)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    return wl.CSR(n, n, ptr, idx, w[at].astype(np.float32))


@pytest.mark.parametrize("n,mids", [(18001, 200), (18001, 700), (40011, 700), (170001, 200), (170001, 5000)])
def test_smallest_distance_found_in_a_listed_chunk(n, mids):
    """A pulled step that brings a row down twice: its first elements make it 150, and 61 comes from the end of the row, which is listed in chunks.  The second time the row
    has been counted already, and 61 is all the same what the next pulled step's rows are cut by: row `r`, at 140, is improved by 61 + 30 and by nothing else."""
    src, hub, r = 0, 33, 55
    mid = 80 + 17 * np.arange(mids)
    far = mid[-1] + 17 * (1 + np.arange(40))
    light = np.where(np.arange(mids) == mids - 1, 1.0, 100.0)
    last = np.where(np.arange(mids) == mids - 1, 60.0, 50.0)
    check_steps(graph(n, [(src, mid, light), (mid, hub, last), (mid[:1], r, 40.0), (hub, r, 30.0), (hub, far, 5.0)]), src)


@pytest.mark.parametrize("mids,early", [(600, 0), (2000, 0), (2000, 80)])
def test_smallest_distance_of_a_pushed_step(mids, early):
    """A pushed step whose frontier, spread over all thread blocks, reaches one vertex from everywhere: the first to lower it counts it, the others bring it further down, and the next step, a pulled one,
    has rows that only the least of these distances improves.  From a listed frontier, from a bitmap, and with so many edges that nothing is listed (`early`: neighbours that were
    reached for nothing, so that nothing else is found)."""
    rng = np.random.default_rng(mids + early)
    reach = 2000000 if early else 100000
    src, hub, rows = 0, 33, 64 + 17 * np.arange(90)
    mid = 2000 + 17 * rng.permutation(mids)
    sinks = reach // 2 - 17 * (1 + np.arange(max(early, 1)))
    out = np.arange(reach // 2, reach, 4)
    edges = [(src, mid, 1.0), (mid, hub, 2.0 + np.arange(mids)), (src, rows, 5.0 + np.arange(90)), (hub, rows, 1.0), (hub, out, 7.0), (src, sinks, 0.0)]
    if early:
        edges.append((mid[:, None], sinks[None, :], 1.0))
    noise = reach + rng.integers(0, reach, (2, reach))                                  # (not reached)
    check_steps(graph(2 * reach, edges + [(noise[0], noise[1], 1.0)]), src, repeats=6)


def test_pulled_steps_of_a_handle_with_many_payload_blocks():
    """A 27-point operator on 21^3 cells, a good part of its elements in blocks with a payload: its steps are pulled from a smaller share of the elements on; noise beside it, not reached, leaves its larger steps
    on both sides of that share."""
    d, far = 21, 21 ** 3
    g, rng = wl.stencil27(d, seed=3), np.random.default_rng(3)
    n = 2 * far
    cells = g.rows(), g.col_idx
    edges = [(cells[1], cells[0], (1 + rng.integers(0, 63, g.nnz)) / 8.0)]
    noise = far + rng.integers(0, far, (2, 250000))
    csr = graph(n, edges + [(noise[0], noise[1], 1.0)])
    h = Handle(csr, B.F32)
    st = h.get_stats()
    assert csr.nnz < 8 * sum(st.class_nnz[1:]) and 2 * sum(st.class_nnz[2:]) < csr.nnz
    h.close()
    for src in (0, d // 2 * (1 + d + d * d)):
        check_steps(csr, src, repeats=2)


@pytest.mark.parametrize("layers,width", [(60, 64), (200, 64), (200, 80)])
def test_many_pulled_steps_of_unit_weights(layers, width):
    """Layers of vertices one behind the other, linked by INLINE elements and by one dense block each, behind a source whose column holds a seventh of the elements: its step is pulled, and so are
    those of the layers, a row's word lowered by its INLINE elements and by the dense block's warp.  (Unit weights: a handle without values.)"""
    rng = np.random.default_rng(layers + width)
    src, first = 0, 48
    u, v = [], []
    for k in range(layers - 1):
        at, per = first + k * width, width // 16
        dense = int(rng.integers(per * per))
        for b in range(per * per):
            r, c = np.divmod(rng.choice(256, 40 if b == dense else 7, replace=False), 16)
            u.append(at + 16 * (b % per) + c)
            v.append(at + width + 16 * (b // per) + r)
    u, v = np.concatenate(u), np.concatenate(v)
    hub = u.size // 6
    far = first + layers * width
    n = far + hub + 5
    u = np.r_[u, np.zeros(width + hub, np.int64)]
    v = np.r_[v, first + np.arange(width), far + np.arange(hub)]
    keys = wl.sorted_unique(v.astype(np.int64) * n + u)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    csr = wl.CSR(n, n, ptr, idx, np.ones(keys.size, np.float32))
    h, A = Handle(csr, B.PATTERN), ref_matrix(csr)
    st = h.get_stats()
    assert sum(st.class_blocks[2:]) == layers - 1 and 2 * sum(st.class_nnz[2:]) < csr.nnz < 10 * (width + hub)
    want = oracle.ref_sssp(A, src)
    assert np.isfinite(want[far - width:far]).any()
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    steps = []
    for path in (B.PATH_AUTO, B.PATH_PUSH, B.PATH_AUTO):
        h.set_opts(force_path=path)
        steps.append(B.db_sssp(h.h, src, dist))
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy().astype(np.float64), want)
    assert steps[0] == steps[1] == steps[2] and steps[0] >= layers
    h.close()


@pytest.mark.parametrize("length", [333, 2000])
@pytest.mark.parametrize("base,step", [(4096.0, 1.0), (-4096.0, 1.0), (300.0, -1.0)])
def test_pulled_steps_of_more_rows_than_lanes(length, base, step):
    """The path of test_many_pulled_steps_in_a_row in a graph with more vertices than the GPU has lanes, where a lane walks a row: distances above zero, below, and such that pass through zero while
    the search goes on (a distance's word is its bits above zero only), in the second launch too."""
    n = length + 107 + 170000
    k = np.arange(length)
    rows = np.r_[1 + k, 2 + k[:-1], length + 1 + np.arange(6)]
    cols = np.r_[np.zeros(length, np.int64), 1 + k[:-1], length + np.arange(6)]
    val = np.r_[base + (step + 1.0) * k, np.full(length - 1, step), np.full(6, 3.0)].astype(np.float32)
    order = np.argsort(rows.astype(np.int64) * n + cols)
    ptr, idx = wl.csr_from_sorted_keys(n, n, (rows.astype(np.int64) * n + cols)[order])
    want = np.full(n, np.inf, np.float32)
    want[0] = 0.0
    want[1:length + 1] = base + step * k
    want[length + 1:length + 7] = base + step * (length - 1) + 3.0 * (1 + np.arange(6))
    h = Handle(wl.CSR(n, n, ptr, idx, val[order]), B.F32)
    dist = torch.empty(n, dtype=torch.float32, device="cuda")
    steps = []
    for path in (B.PATH_AUTO, B.PATH_PUSH, B.PATH_AUTO):
        h.set_opts(force_path=path)
        steps.append(B.db_sssp(h.h, 0, dist))
        torch.cuda.synchronize()
        assert np.array_equal(dist.cpu().numpy(), want)
    assert steps[0] == steps[1] == steps[2] and steps[0] > length
    h.close()


def test_pulled_steps_of_a_large_handle_with_many_payload_blocks():
    """A 27-point operator on 55^3 cells, more rows than the GPU has lanes: its steps are pulled from the larger share of the elements on, those behind them from an eighth of the rows' number of edges at most."""
    d = 55
    g, rng = wl.stencil27(d, seed=3), np.random.default_rng(3)
    cells = g.rows(), g.col_idx
    csr = graph(g.n, [(cells[1], cells[0], (1 + rng.integers(0, 63, g.nnz)) / 8.0)])
    h = Handle(csr, B.F32)
    st = h.get_stats()
    assert csr.nnz < 8 * sum(st.class_nnz[1:]) and 2 * sum(st.class_nnz[2:]) < csr.nnz
    h.close()
    check_steps(csr, d // 2 * (1 + d + d * d))
