"""GPU parity of db_bfs: levels bit-identical to the queue BFS of the oracle, for forced push,
forced pull and the per-level automatic switch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, ref_matrix, DEV

pytestmark = pytest.mark.gpu
PATHS = [B.PATH_AUTO, B.PATH_PUSH, B.PATH_PULL]


def bfs(h, src):
    levels = torch.full((h.csr.n,), -5, dtype=torch.int32, device=DEV)
    B.db_bfs(h.h, int(src), levels)
    torch.cuda.synchronize()
    return levels.cpu().numpy()


def graph_from_edges(n, edges):
    a = np.zeros((n, n), dtype=np.float32)
    for u, v in edges:
        a[v, u] = 1.0                      # stored A[v][u] is the edge u -> v
    return wl.csr_from_dense(a)


GRAPHS = [
    ("rmat12", lambda: wl.rmat(12, 16, seed=3, values=False, symmetrise=True)),
    ("rmat14", lambda: wl.rmat(14, 16, seed=4, values=False, symmetrise=True)),
    ("grid20", lambda: wl.stencil27(20, values=False)),
    ("directed_random", lambda: wl.random_sparse(3000, 3000, 9000, 5, values=False)),
    ("ragged_directed", lambda: wl.random_sparse(1000 + 7, 1000 + 7, 4000, 6, values=False)),
]


@pytest.mark.parametrize("name,make", GRAPHS, ids=[g[0] for g in GRAPHS])
@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("inline_max,no_index", [(31, 0), (3, 0), (31, 1)], ids=["inline", "coo_lists", "no_row_index"])
def test_levels_bit_exact(name, make, path, inline_max, no_index):
    g = make()
    o = B.default_create_opts()
    o.inline_max = inline_max            # 3: blocks of 4..31 entries become packed coordinate lists
    o.no_bfs_index = no_index            # 1: pull levels walk the row-block segments
    h = Handle(g, B.PATTERN, opts=o)
    h.set_opts(force_path=path)
    A = ref_matrix(g)
    deg = np.diff(g.row_ptr)
    srcs = [0, int(np.argmax(deg)), g.n - 1] + [int(s) for s in wl.bfs_sources(g, 3, seed=9)]
    for s in srcs:
        want = oracle.ref_bfs(A, s)
        got = bfs(h, s)
        assert np.array_equal(got, want), f"source {s}"
        st = h.get_stats()
        assert st.bfs_reached == int((want >= 0).sum())
        assert st.bfs_levels == int(want.max()) + 1     # the last expansion finds nothing new
    h.close()


def test_small_graphs_with_known_levels():
    n = 50
    path = graph_from_edges(n, [(i, i + 1) for i in range(n - 1)] + [(i + 1, i) for i in range(n - 1)])
    h = Handle(path, B.PATTERN)
    for p in PATHS:
        h.set_opts(force_path=p)
        assert bfs(h, 0).tolist() == list(range(n))
        assert bfs(h, 20).tolist() == [abs(i - 20) for i in range(n)]
    h.close()
    cyc = graph_from_edges(3, [(0, 1), (1, 2), (2, 0)])     # pins the edge orientation
    h = Handle(cyc, B.PATTERN)
    for p in PATHS:
        h.set_opts(force_path=p)
        assert bfs(h, 0).tolist() == [0, 1, 2]
    h.close()
    two = graph_from_edges(7, [(0, i) for i in range(1, 5)] + [(i, 0) for i in range(1, 5)] + [(5, 6), (6, 5)])
    h = Handle(two, B.PATTERN)
    for p in PATHS:
        h.set_opts(force_path=p)
        assert bfs(h, 0).tolist() == [0, 1, 1, 1, 1, -1, -1]
        assert bfs(h, 5).tolist() == [-1, -1, -1, -1, -1, 0, 1]
    h.close()


def test_isolated_source_and_bad_arguments():
    g = graph_from_edges(40, [(1, 2), (2, 1)])
    h = Handle(g, B.PATTERN)
    lv = bfs(h, 0)
    assert lv[0] == 0 and (lv[1:] == -1).all()
    assert h.get_stats().bfs_levels == 1 and h.get_stats().bfs_reached == 1
    levels = torch.empty(40, dtype=torch.int32, device=DEV)
    for bad in (-1, 40):
        with pytest.raises(B.DbSpmspvError) as e:
            B.db_bfs(h.h, bad, levels)
        assert e.value.status == B.ERR_INVALID_ARG
    h.close()
    rect = Handle(wl.random_sparse(30, 40, 100, 1, values=False), B.PATTERN)
    with pytest.raises(B.DbSpmspvError) as e:
        B.db_bfs(rect.h, 0, levels)
    assert e.value.status == B.ERR_UNSUPPORTED
    rect.close()


def test_chebyshev_closed_form_and_valued_handle():
    """On the 27-point grid graph level(v) = max(|dx|,|dy|,|dz|); a valued (fp32) handle gives
    the same levels as the pattern one; an SpMSpV call after a BFS on the same handle is clean."""
    d = 32
    g = wl.stencil27(d, seed=2)
    h = Handle(g, B.F32)
    ar = np.arange(d)
    z, y, x = np.meshgrid(ar, ar, ar, indexing="ij")
    sx, sy, sz = 3, 30, 17
    want = np.maximum(np.maximum(abs(x - sx), abs(y - sy)), abs(z - sz)).reshape(-1).astype(np.int32)
    for p in PATHS:
        h.set_opts(force_path=p)
        assert np.array_equal(bfs(h, sx + d * (sy + d * sz)), want)
    st = h.get_stats()
    assert st.bfs_levels == want.max() + 1        # the last expansion finds nothing new
    from gpu_util import check_against_oracle
    xs = wl.clustered_x(g.n, 8)
    h.set_opts()
    check_against_oracle(h.run(xs), oracle.ref_pull(ref_matrix(g), xs.idx, xs.val))
    h.close()


def test_auto_switches_direction_across_levels():
    g = wl.rmat(14, 16, seed=4, values=False, symmetrise=True)
    h = Handle(g, B.PATTERN)
    h.set_opts(th3_bfs=0.01)
    src = int(wl.bfs_sources(g, 1, seed=9)[0])
    bfs(h, src)
    st = h.get_stats()
    paths = list(st.bfs_level_path[:st.bfs_levels])
    nz = list(st.bfs_level_nzblk[:st.bfs_levels])
    nblk = (g.n + 15) // 16
    for p, k in zip(paths, nz):
        assert p == (B.PATH_PUSH if np.float32(k) / np.float32(nblk) < np.float32(0.01) else B.PATH_PULL)
    assert B.PATH_PUSH in paths and B.PATH_PULL in paths
    h.close()


def test_hub_column_goes_through_the_hub_list():
    """A star with 12,000 leaves: the centre's column holds more INLINE elements than the hub
    threshold, so its push is not cut into tasks but strided over by all warps."""
    n = 12001
    rows = np.r_[np.zeros(n - 1, np.int64), np.arange(1, n)]
    cols = np.r_[np.arange(1, n), np.zeros(n - 1, np.int64)]
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    row_ptr = np.r_[0, np.cumsum(np.bincount(rows, minlength=n))].astype(np.int64)
    g = wl.CSR(n, n, row_ptr, cols.astype(np.int32), None)
    A = ref_matrix(g)
    for path in (B.PATH_PUSH, B.PATH_AUTO):
        h = Handle(g, B.PATTERN)
        h.set_opts(force_path=path)
        for s in (5, 0, n - 1):
            assert np.array_equal(bfs(h, s), oracle.ref_bfs(A, s)), f"source {s}"
        h.close()


@pytest.mark.parametrize("n", [700, 17000, 70001])
@pytest.mark.parametrize("fan", [15 * 32, 16 * 32, 16 * 32 + 1, 17 * 32])
def test_small_push_levels(n, fan):
    """A level of 15 to 17 warp steps, with and without a successor that is surely a push: vertex 3 reaches `fan` vertices,
    each of them one or two of the others."""
    rng = np.random.default_rng(fan)
    first = rng.permutation(np.arange(4, n))[:min(fan, n - 10)]
    u = np.r_[np.full(first.size, 3), np.repeat(first, 2), [0]]
    v = np.r_[first, rng.integers(4, n, 2 * first.size), [3]]
    keys = wl.sorted_unique(v.astype(np.int64) * n + u)
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    for path in PATHS:
        h.set_opts(force_path=path)
        for s in (0, 3, int(first[0])):
            want = oracle.ref_bfs(A, s)
            assert np.array_equal(bfs(h, s), want)
            assert h.get_stats().bfs_reached == int((want >= 0).sum())
    h.close()


def test_push_levels_past_the_step_limit():
    """Forced pushes whose largest level has more than 16384 warp steps (1.9 M entries), and the automatic search beside them."""
    g = wl.rmat(16, 16, seed=12, values=False, symmetrise=True)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    for path in (B.PATH_PUSH, B.PATH_AUTO):
        h.set_opts(force_path=path)
        for s in [int(np.argmax(np.diff(g.row_ptr)))] + [int(q) for q in wl.bfs_sources(g, 3, seed=2)]:
            want = oracle.ref_bfs(A, s)
            assert np.array_equal(bfs(h, s), want)
            assert h.get_stats().bfs_reached == int((want >= 0).sum())
    h.close()


@pytest.mark.parametrize("n", [65535, 65537, 70001, 70016])
def test_large_levels_of_ragged_graphs(n):
    """Push levels past the step limit (levels, visited and counts come from a pass over the masks behind them) and pull levels in which most rows end at their
    first element, on graphs whose last mask word is not full; the levels start at an address that is not a multiple of 16 bytes."""
    rng = np.random.default_rng(n)
    hub = rng.integers(0, 64, 4 * n)
    u, v = np.r_[hub, rng.integers(0, n, 12 * n)], rng.integers(0, n, 16 * n)
    keep = u != v
    keys = wl.sorted_unique(np.r_[u[keep] * n + v[keep], v[keep] * n + u[keep]].astype(np.int64))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    levels = torch.empty(n + 1, dtype=torch.int32, device="cuda")[1:]
    for src in (n - 1, 5):
        want = oracle.ref_bfs(A, src)
        for path in PATHS:
            h.set_opts(force_path=path)
            levels.fill_(7)
            B.db_bfs(h.h, src, levels)
            torch.cuda.synchronize()
            assert np.array_equal(levels.cpu().numpy(), want)
            assert h.get_stats().bfs_reached == int((want >= 0).sum())
    h.close()


@pytest.mark.parametrize("delta", [0, 1, 33, 5001])
def test_levels_on_both_sides_of_the_large_graph_rule(delta):
    """Graphs of at most / more than four mask words per warp of the grid: from there on a pull looks at the first element of every row before its run,
    and pushed frontiers are counted by elements.  Two hubs (pushes of many elements), sparse random edges, a path that ends in the last word."""
    n = torch.cuda.get_device_properties(0).multi_processor_count * 32 * 4 * 32 + delta
    rng = np.random.default_rng(delta)
    hub = rng.integers(0, 2, n) * 7
    u, v = np.r_[hub, rng.integers(0, n, 2 * n), np.arange(n - 12, n - 1)], np.r_[rng.integers(0, n, 3 * n), np.arange(n - 11, n)]
    keep = u != v
    keys = wl.sorted_unique(np.r_[u[keep] * n + v[keep], v[keep] * n + u[keep]].astype(np.int64))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    for src in (n - 1, 7):
        want = oracle.ref_bfs(A, src)
        for path in PATHS:
            h.set_opts(force_path=path)
            assert np.array_equal(bfs(h, src), want)
            st = h.get_stats()
            assert st.bfs_reached == int((want >= 0).sum()) and st.bfs_levels == int(want.max()) + 1
    h.close()


@pytest.mark.parametrize("fan", [1, 1023, 1024, 1025, 6000])
def test_listed_and_unlisted_frontiers(fan):
    """Frontiers at the length up to which they are kept as a list of vertices (1024), in turn with longer and shorter ones: the source reaches `fan` vertices, they reach a third of that
    and one vertex whose column is long, then single vertices; dense blocks (with a payload) among the first ones; a part that is not reached keeps the levels a small share of the graph."""
    n = 40011
    rng = np.random.default_rng(fan)
    a = 16 + np.arange(fan)
    b = 8000 + np.arange(max(1, fan // 3))
    u = [np.full(fan, 3), a, np.full(1, a[0]), np.full(700, 20000), [20001, 20002, 20003], np.repeat(np.arange(16, 48), 24), rng.integers(22000, n, 100000)]
    v = [a, b[rng.integers(0, b.size, fan)], [20000], 20001 + np.arange(700), [21000, 21001, 21002], np.tile(np.arange(30000, 30024), 32), rng.integers(22000, n, 100000)]
    keys = wl.sorted_unique(np.concatenate(v).astype(np.int64) * n + np.concatenate(u))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    for src in (3, 20000, int(a[-1])):
        want = oracle.ref_bfs(A, src)
        for path in PATHS:
            h.set_opts(force_path=path)
            assert np.array_equal(bfs(h, src), want)
            st = h.get_stats()
            assert st.bfs_reached == int((want >= 0).sum()) and st.bfs_levels == int(want.max()) + 1
    h.close()


@pytest.mark.parametrize("n", [170001, 178001])
def test_short_frontier_of_many_elements(n):
    """Three vertices that reach all others: 510,000 and 534,000 elements, on both sides of what a listed frontier is pushed from its list with (524,288)."""
    hubs = np.array([5, 70000, n - 1])
    u = np.r_[np.full(3, 9), np.repeat(hubs, n)]
    v = np.r_[hubs, np.tile(np.arange(n), 3)]
    keep = u != v
    keys = wl.sorted_unique(v[keep].astype(np.int64) * n + u[keep])
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    for src in (9, 70000):
        want = oracle.ref_bfs(A, src)
        for path in PATHS:
            h.set_opts(force_path=path)
            assert np.array_equal(bfs(h, src), want)
            assert h.get_stats().bfs_reached == n
    h.close()


def test_pulled_row_blocks_by_their_entries_with_a_payload():
    """A pulled level takes the two row blocks of a mask word side by side while both have at most 16 entries with a payload: every pair of counts around that and around a warp's 32.  (These rows have
    no other parents; a dense block has 40 elements, and one row without any.)"""
    counts = [0, 1, 15, 16, 17, 32, 33, 65]
    pairs = [(a, b) for a in counts for b in counts]
    n = 60000 + 5
    rng = np.random.default_rng(5)
    rows, cols = [], []
    for w, pair in enumerate(pairs):
        for half, count in enumerate(pair):
            for cb in np.sort(rng.choice(np.arange(400, 2400), count, replace=False)):          # dense blocks, one row of each left out
                r, c = np.divmod(np.setdiff1d(np.arange(256), 16 * (cb % 16) + np.arange(16))[rng.choice(240, 40, replace=False)], 16)
                rows.append(16 * (2 * w + half) + r)
                cols.append(16 * cb + c)
    rows += [rng.integers(2048, n, 300000), 40000 + np.arange(300)]
    cols += [40000 + rng.integers(0, n - 40000, 300000), np.full(300, 7)]
    keys = wl.sorted_unique(np.concatenate(rows).astype(np.int64) * n + np.concatenate(cols))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    g = wl.CSR(n, n, ptr, idx, None)
    h, A = Handle(g, B.PATTERN), ref_matrix(g)
    st = h.get_stats()
    assert st.bfs_index_bytes > 0 and sum(st.class_blocks[2:]) == sum(a + b for a, b in pairs)
    for src in (7, 16 * 400 + 3, 40007, n - 1):
        want = oracle.ref_bfs(A, src)
        for path in PATHS:
            h.set_opts(force_path=path)
            assert np.array_equal(bfs(h, src), want)
    h.close()
