"""Performance cases of the library: the calls a user's program makes, over the range of sizes it
makes them at.  Every input is made on the GPU from a seed; matrices follow the shapes of the
benchmark's configurations (uniform rows, R-MAT graphs, the 27-point stencil, pruned layers).

Five kinds of call are covered:
  spmspv   y = A x, fp32, (+, *): sparse x in, sorted sparse y out (dbspmspv_run)
  masked   one Boolean step of a graph traversal with the visited rows masked out (dbspmspv_run_masked)
  bfs      breadth-first levels from one source (db_bfs)
  sssp     shortest-path distances from one source (db_sssp)
  decode   y = W x for one activation vector or a small batch, bf16 weights (dbspmspv_decode / _batch)
"""
import math
from statistics import NormalDist

import torch

from paper_2608_16308_b200 import binding as B

DEV = "cuda"
RMAT_PROBS = (0.57, 0.19, 0.19, 0.05)
EDGE_FACTOR = 16


def listed():
    return [
        # one product on a small matrix, x 1 % full: the call's latency (a step of an iterative
        # solver on a coarse grid, a rule lookup)
        {"name": "uniform16k_x1pct", "kind": "spmspv", "matrix": "uniform", "n": 16384, "x": 0.01, "relabel": False},
        # the input-sparsity sweep on a power-law matrix with a million rows: a handful of listed
        # columns (local graph queries, seeded random walks), ordinary frontiers, and half of all
        # columns listed (late iterations of a rank or label propagation)
        {"name": "rmat20_x1e-4", "kind": "spmspv", "matrix": "rmat", "n": 1 << 20, "x": 1e-4, "relabel": False},
        {"name": "rmat20_x1pct", "kind": "spmspv", "matrix": "rmat", "n": 1 << 20, "x": 0.01, "relabel": False},
        {"name": "rmat20_x10pct", "kind": "spmspv", "matrix": "rmat", "n": 1 << 20, "x": 0.1, "relabel": False},
        {"name": "rmat20_x50pct", "kind": "spmspv", "matrix": "rmat", "n": 1 << 20, "x": 0.5, "relabel": False},
        # a discretised operator applied to a vector with local support (runs of 64 entries)
        {"name": "stencil160_x5pct", "kind": "spmspv", "matrix": "stencil", "n": 160, "x": 0.05, "relabel": False},
        # one traversal step driven by the caller: Boolean product, visited rows masked out, an odd
        # number of vertices in scattered order
        {"name": "masked300007_x3pct", "kind": "masked", "n": 300007, "x": 0.03, "relabel": True},
        # a whole breadth-first search and a whole shortest-path search
        {"name": "bfs_rmat22", "kind": "bfs", "n": 1 << 22, "relabel": False},
        {"name": "sssp_rmat20", "kind": "sssp", "n": 1 << 20, "relabel": False},
        # one token through a pruned linear layer, activations 30 % and 10 % nonzero; eight tokens
        {"name": "decode_12288x4096_a30", "kind": "decode", "m": 12288, "n": 4096, "prune": 0.5, "active": 0.3, "batch": 1},
        {"name": "decode_4096x11008_a10", "kind": "decode", "m": 4096, "n": 11008, "prune": 0.7, "active": 0.1, "batch": 1},
        {"name": "decode_11008x4096_b8", "kind": "decode", "m": 11008, "n": 4096, "prune": 0.5, "active": 0.3, "batch": 8},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["spmspv", "spmspv", "spmspv", "masked", "bfs", "sssp", "decode", "decode"])
    if kind == "spmspv":
        matrix = rng.choice(["uniform", "rmat", "rmat", "stencil"])
        n = int(_log_uniform(rng, 24, 160.99)) if matrix == "stencil" else int(_log_uniform(rng, 4096, 1 << 20))
        return {"kind": kind, "matrix": matrix, "n": n, "x": round(_log_uniform(rng, 1e-5, 0.5), 7),
                "relabel": matrix == "rmat" and rng.random() < 0.5}
    if kind == "masked":
        return {"kind": kind, "n": int(_log_uniform(rng, 16384, 1 << 20)), "x": round(_log_uniform(rng, 1e-5, 0.3), 7),
                "relabel": rng.random() < 0.5}
    if kind == "bfs":
        return {"kind": kind, "n": int(_log_uniform(rng, 16384, 1 << 22)), "relabel": rng.random() < 0.5}
    if kind == "sssp":
        return {"kind": kind, "n": int(_log_uniform(rng, 16384, 1 << 20)), "relabel": rng.random() < 0.5}
    m = int(_log_uniform(rng, 1024, 12288))
    n = int(_log_uniform(rng, 1024, min(12288, 12288 * 4096 / m)))
    return {"kind": kind, "m": m, "n": n, "prune": rng.choice([0.5, 0.6, 0.7]), "active": round(rng.uniform(0.05, 0.5), 3),
            "batch": rng.choice([1, 1, 2, 3, 4, 6, 8])}


# ----------------------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------------------
class _Handle:
    """Owns a library handle for as long as the state lives."""

    def __init__(self, value):
        self.value = value

    def __del__(self):
        if self.value and B is not None:
            B.dbspmspv_destroy(self.value)
            self.value = None


def _uniform(gen, n, lo, hi):
    return torch.rand(n, generator=gen, device=DEV) * (hi - lo) + lo


def _csr(m, n, keys):
    """Sorted unique keys row * n + col -> row pointers (int64) and columns (int32)."""
    rows = torch.div(keys, n, rounding_mode="floor")
    cols = (keys - rows * n).to(torch.int32)
    ptr = torch.searchsorted(rows, torch.arange(m + 1, device=DEV, dtype=torch.int64))
    return ptr, cols


def _sorted_unique(keys):
    keys = torch.sort(keys).values
    keep = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
    keep[1:] = keys[1:] != keys[:-1]
    return keys[keep]


def _rmat(gen, n, relabel, symmetric):
    """R-MAT on n vertices (a power of two, or the next one's numbering scaled down to n), duplicates merged."""
    scale = max(1, (n - 1).bit_length())
    edges = EDGE_FACTOR * n
    row = torch.zeros(edges, dtype=torch.int64, device=DEV)
    col = torch.zeros(edges, dtype=torch.int64, device=DEV)
    a, b, c, _ = RMAT_PROBS
    for _ in range(scale):
        u = torch.rand(edges, generator=gen, device=DEV)
        down = u >= a + b
        right = ((u >= a) & ~down) | (u >= a + b + c)
        row = row * 2 + down
        col = col * 2 + right
    if n != 1 << scale:
        row = (row * n) >> scale
        col = (col * n) >> scale
    if relabel:
        perm = torch.randperm(n, generator=gen, device=DEV)
        row, col = perm[row], perm[col]
    if symmetric:
        keep = row != col
        row, col = row[keep], col[keep]
        row, col = torch.cat([row, col]), torch.cat([col, row])
    return _csr(n, n, _sorted_unique(row * n + col))


def _stencil(gen, d):
    """27-point operator on a d^3 grid: off-diagonals U(0.5, 1.5), diagonal 27."""
    n = d ** 3
    i = torch.arange(n, device=DEV)
    x, y, z = i % d, torch.div(i, d, rounding_mode="floor") % d, torch.div(i, d * d, rounding_mode="floor")
    cols = torch.empty((n, 27), dtype=torch.int32, device=DEV)
    ok = torch.empty((n, 27), dtype=torch.bool, device=DEV)
    k = 0
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                ok[:, k] = (z + dz >= 0) & (z + dz < d) & (y + dy >= 0) & (y + dy < d) & (x + dx >= 0) & (x + dx < d)
                cols[:, k] = i + dx + d * (dy + d * dz)
                k += 1
    counts = ok.sum(dim=1)
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=ptr[1:])
    col = cols[ok]
    val = _uniform(gen, col.numel(), 0.5, 1.5)
    diagonal = torch.zeros((n, 27), dtype=torch.bool, device=DEV)
    diagonal[:, 13] = True
    val[diagonal[ok]] = 27.0
    return ptr, col, val


def _sparse_x(gen, n, count, clustered):
    if clustered:      # runs of 64 consecutive indices, none overlapping another, at unaligned starts
        slots = max(1, n // 80)
        runs = min(slots, max(1, count // 64))
        at = torch.randperm(slots, generator=gen, device=DEV)[:runs] * 80
        at = at + torch.randint(0, 17, (runs,), generator=gen, device=DEV)
        idx = (at[:, None] + torch.arange(64, device=DEV)).reshape(-1).to(torch.int32)
    else:
        idx = torch.randperm(n, generator=gen, device=DEV)[:count].to(torch.int32)
    val = _uniform(gen, idx.numel(), -1.0, 1.0)
    val[val == 0] = 0.5
    return idx, val


def _count(case, n):
    return max(1, int(n * case["x"] + 0.5))


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    if kind == "decode":
        m, n = case["m"], case["n"]
        # magnitude-pruned N(0, 0.02) weights; activations ReLU(N(mu, 1)) with the given share above zero
        w = torch.randn((m, n), generator=gen, device=DEV) * 0.02
        keep = w.abs() >= 0.02 * NormalDist().inv_cdf((1 + case["prune"]) / 2)
        ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(keep.sum(dim=1), 0, out=ptr[1:])
        col = keep.nonzero()[:, 1].to(torch.int32)
        val = w[keep].to(torch.bfloat16)
        mu = -NormalDist().inv_cdf(1 - case["active"])
        x = torch.relu(torch.randn((case["batch"], n), generator=gen, device=DEV) + mu).to(torch.bfloat16)
        h = _Handle(B.dbspmspv_create_csr(m, n, col.numel(), ptr, col, val, B.BF16))
        return {"kind": kind, "h": h, "x": x, "y": torch.zeros((case["batch"], m), device=DEV), "m": m, "n": n, "batch": case["batch"]}
    if kind in ("bfs", "sssp"):
        n = case["n"]
        ptr, col = _rmat(gen, n, case["relabel"], True)
        # a source with at least one edge, uniformly among them
        with_edges = (ptr[1:] > ptr[:-1]).nonzero()[:, 0]
        src = int(with_edges[int(torch.randint(0, with_edges.numel(), (1,), generator=gen, device=DEV))])
        if kind == "bfs":
            h = _Handle(B.dbspmspv_create_csr(n, n, col.numel(), ptr, col, None, B.PATTERN))
            out = torch.empty(n, dtype=torch.int32, device=DEV)
        else:
            h = _Handle(B.dbspmspv_create_csr(n, n, col.numel(), ptr, col, _uniform(gen, col.numel(), 0.05, 1.05), B.F32))
            out = torch.empty(n, device=DEV)
        return {"kind": kind, "h": h, "src": src, "out": out}
    if kind == "masked":
        n = m = case["n"]
        ptr, col = _rmat(gen, n, case["relabel"], True)
        h = _Handle(B.dbspmspv_create_csr(n, n, col.numel(), ptr, col, None, B.PATTERN))
        idx, val = _sparse_x(gen, n, _count(case, n), False)
        # the visited set: a tenth of the vertices and the frontier itself, one bit per row
        bits = torch.rand(n, generator=gen, device=DEV) < 0.1
        bits[idx.long()] = True
        words = (n + 31) // 32
        padded = torch.zeros(words * 32, dtype=torch.int64, device=DEV)
        padded[:n] = bits
        visited = (padded.view(words, 32) << torch.arange(32, device=DEV)).sum(dim=1).to(torch.int32)
        return _sparse_state(kind, h, m, idx, None, visited)
    n = case["n"]
    if case["matrix"] == "stencil":
        ptr, col, val = _stencil(gen, n)
        n = n ** 3
    elif case["matrix"] == "rmat":
        ptr, col = _rmat(gen, n, case["relabel"], False)
        val = _uniform(gen, col.numel(), -1.0, 1.0)
    else:
        col = torch.sort(torch.randint(0, n, (n, 8), generator=gen, device=DEV), dim=1).values.reshape(-1).to(torch.int32)
        ptr = torch.arange(0, 8 * n + 1, 8, dtype=torch.int64, device=DEV)
        val = _uniform(gen, col.numel(), -1.0, 1.0)
    h = _Handle(B.dbspmspv_create_csr(n, n, col.numel(), ptr, col, val, B.F32))
    idx, xv = _sparse_x(gen, n, _count(case, n), case["matrix"] == "stencil")
    return _sparse_state(kind, h, n, idx, xv, None)


def _sparse_state(kind, h, m, idx, val, visited):
    return {"kind": kind, "h": h, "m": m, "x_idx": idx, "x_val": val, "nnz_x": idx.numel(), "visited": visited,
            "y_idx": torch.zeros(m, dtype=torch.int32, device=DEV), "y_val": torch.zeros(m, device=DEV),
            "y_nnz": torch.zeros(1, dtype=torch.int32, device=DEV)}


def run(s):
    kind = s["kind"]
    if kind == "spmspv":
        B.dbspmspv_run(s["h"].value, s["x_idx"], s["x_val"], s["nnz_x"], B.PLUS_TIMES, s["y_idx"], s["y_val"], s["m"], s["y_nnz"])
        return s["y_idx"], s["y_val"], s["y_nnz"]
    if kind == "masked":
        B.dbspmspv_run_masked(s["h"].value, s["x_idx"], None, s["nnz_x"], B.OR_AND, s["visited"], 1, s["y_idx"], None, s["m"], s["y_nnz"])
        return s["y_idx"], s["y_nnz"]
    if kind == "bfs":
        B.db_bfs(s["h"].value, s["src"], s["out"])
        return s["out"]
    if kind == "sssp":
        steps = B.db_sssp(s["h"].value, s["src"], s["out"])
        return s["out"], steps
    if s["batch"] == 1:
        B.dbspmspv_decode(s["h"].value, s["x"], s["y"])
    else:
        B.dbspmspv_decode_batch(s["h"].value, s["x"], s["n"], s["y"], s["m"], s["batch"])
    return s["y"]


# ----------------------------------------------------------------------------------------
# Work
# ----------------------------------------------------------------------------------------
def _rmat_rows_hit(n, share, factor):
    """Expected rows with at least one listed column: rows by their number of one bits, degrees Poisson."""
    scale = max(1, (n - 1).bit_length())
    up, down = RMAT_PROBS[0] + RMAT_PROBS[1], RMAT_PROBS[2] + RMAT_PROBS[3]
    hit = 0.0
    for k in range(scale + 1):
        degree = factor * n * up ** (scale - k) * down ** k * (1 << scale) / n
        hit += math.comb(scale, k) * (1 - math.exp(-degree * share))
    return hit * n / (1 << scale)


def work(case):
    """Bytes and operations of one pass that no implementation does without (expected values: they
    follow from the sizes and the distributions, not from one seed's matrix)."""
    kind = case["kind"]
    if kind == "decode":
        # the surviving weights of the columns that some vector reaches, and their positions (a bit each)
        m, n, b = case["m"], case["n"], case["batch"]
        reached = 1 - (1 - case["active"]) ** b
        return {"bytes": m * n * reached * (2 * (1 - case["prune"]) + 1 / 8) + b * (2 * n + 4 * m),
                "flops": 2.0 * m * n * (1 - case["prune"]) * case["active"] * b}
    if kind == "bfs":
        # every level is written; a vertex that is reached has its row's place and one edge read
        return {"bytes": 12.0 * case["n"], "flops": 0.0}
    if kind == "sssp":
        # every edge is relaxed at least once (index and weight); every distance is written
        edges = 2.0 * EDGE_FACTOR * case["n"]
        return {"bytes": 8.0 * edges + 4.0 * case["n"], "flops": edges}
    if kind == "masked":
        n = case["n"]
        x = _count(case, n)
        edges = 2.0 * EDGE_FACTOR * n * x / n
        return {"bytes": 12.0 * x + 4.0 * edges + n / 8 + 4 * 0.9 * _rmat_rows_hit(n, x / n, 2 * EDGE_FACTOR), "flops": edges}
    # the listed columns: pointers, row indices and values; x; y (index and value)
    n = case["n"]
    if case["matrix"] == "stencil":
        n = n ** 3
        x = _count(case, n)
        products, rows = 27.0 * x, min(float(n), x * 9.0 * 66 / 64)
    else:
        x = _count(case, n)
        products = (EDGE_FACTOR if case["matrix"] == "rmat" else 8.0) * x
        rows = _rmat_rows_hit(n, x / n, EDGE_FACTOR) if case["matrix"] == "rmat" else n * (1 - (1 - x / n) ** 8)
    return {"bytes": 16.0 * x + 8.0 * products + 8.0 * rows, "flops": 2.0 * products}


def tolerance(case):
    # levels, masked index sets: whole numbers.  Distances are exact minima of sums made in path
    # order.  Products: fp32 sums in an order of the implementation's choice (bf16 products are exact in fp32).
    if case["kind"] in ("bfs", "masked"):
        return "exact"
    if case["kind"] == "sssp":
        return {"rel": 1e-6}
    return {"rel": 1e-5}
