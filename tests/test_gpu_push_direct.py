"""The direct push of hypersparse handles and the finishing kernel behind it: columns at the limit of a listed chunk, blocks with a
payload, a hub row, tiles of the finishing kernel and groups of them, x taken from its list and from the masks."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, check_against_oracle, ref_matrix

pytestmark = pytest.mark.gpu


def matrix(m, n, seed):
    """Columns of 127 .. 1025 elements, row 33 full, four full blocks, sparse noise; products down to 2^-122, zeros of both signs."""
    bg = wl.random_sparse(m, n, min(3 * m, 200000), seed)
    rng = np.random.default_rng(seed)
    rows, cols = [bg.rows(), np.full(n, 33)], [bg.col_idx, np.arange(n)]
    for c, k in ((3, 127), (4, 128), (21, 129), (300, 257), (n - 1, 1025)):
        rows.append(rng.choice(m, k, replace=False))
        cols.append(np.full(k, c))
    for rb, cb in ((0, 0), (m // 16 - 1, 0), (7, 1), (9, n // 16 - 1)):
        r, c = np.mgrid[16 * rb:16 * rb + 16, 16 * cb:16 * cb + 16]
        rows.append(r.ravel())
        cols.append(c.ravel())
    keys = wl.sorted_unique(np.concatenate(rows).astype(np.int64) * n + np.concatenate(cols))
    ptr, idx = wl.csr_from_sorted_keys(m, n, keys)
    val = rng.choice(np.float32([1.5, -0.75, 0.125, 3.0, 0.0, -0.0, 2.0 ** -60, -2.0 ** -62]), keys.size).astype(np.float32)
    return wl.CSR(m, n, ptr, idx, val)


@pytest.mark.parametrize("m", [2047, 2048, 2049, 33 * 2048 + 5,            # a tile of rows; more than a group of 32 tiles
                               2048 * 1185, 2048 * 2400 + 7])               # two and three tiles per thread block
@pytest.mark.parametrize("dtype", [B.F32, B.BF16, B.PATTERN])
def test_direct_push(m, dtype):
    n = 40009
    csr = matrix(m, n, 5)
    h = Handle(csr, dtype)
    assert h.stats.n_hub_row_blocks > 0
    A = ref_matrix(csr, bf16=dtype == B.BF16)
    P = oracle.RefMatrix(csr.m, csr.n, csr.row_ptr, csr.col_idx, None)
    rng = np.random.default_rng(m)
    always = np.int32([3, 4, 21, 300, n - 1])
    lists = [always, np.arange(n // 8, dtype=np.int32)]                 # the list form; enough entries for a pull, too few blocks (masks)
    lists += [np.unique(np.r_[always, rng.choice(n, k)]).astype(np.int32) for k in (40, 3000, 6000)]
    for idx in lists:
        x = wl.SparseVec(n, idx, rng.choice(np.float32([1.0, -2.0, 0.5, -0.0, 2.0 ** -60]), idx.size).astype(np.float32))
        for semiring in (B.OR_AND, B.MIN_PLUS) if dtype == B.PATTERN else (B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS):
            h.set_opts(no_small_call=1)
            got = h.run(x, semiring=semiring)
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(P if dtype == B.PATTERN else A, x.idx, x.val)
                assert np.array_equal(got[0], wi) and np.array_equal(got[1], wv.astype(np.float32))
            else:
                check_against_oracle(got, oracle.ref_pull(P if dtype == B.PATTERN else A, x.idx, x.val), boolean=semiring == B.OR_AND)
            assert h.get_stats().last_path == B.PATH_PUSH
    h.close()


@pytest.mark.parametrize("dtype", [B.F32, B.PATTERN])
def test_long_x_on_a_handle_rich_in_payload(dtype):
    csr = wl.stencil27(40, seed=3)
    h = Handle(csr, dtype)
    P = oracle.RefMatrix(csr.m, csr.n, csr.row_ptr, csr.col_idx, None)
    for lo, hi in ((0, csr.n // 8), (17, csr.n // 2), (0, csr.n)):          # the last one pulls
        idx = np.arange(lo, hi, dtype=np.int32)
        x = wl.SparseVec(csr.n, idx, np.random.default_rng(hi).choice(np.float32([1.0, -2.0, 0.5, -0.0]), idx.size).astype(np.float32))
        for semiring in ([B.OR_AND] if dtype == B.PATTERN else [B.PLUS_TIMES, B.OR_AND]):
            want = oracle.ref_pull(P if dtype == B.PATTERN else ref_matrix(csr), x.idx, x.val)
            check_against_oracle(h.run(x, semiring=semiring), want, boolean=semiring == B.OR_AND)
            assert h.get_stats().last_path == (B.PATH_PULL if hi - lo == csr.n else B.PATH_PUSH)
    h.close()


def blocks_and_noise(n, seed):
    """A quarter of the elements in blocks with a payload -- dense, a few full rows, a few full columns, scattered -- of 32 to 256
    elements each, the rest single."""
    rng = np.random.default_rng(seed)
    bg = wl.random_sparse(n, n, 4 * n, seed)
    rows, cols = [bg.rows()], [bg.col_idx]
    for k in range(2200):
        rb, cb = rng.integers(0, n // 16, 2)
        full = np.zeros((16, 16), bool)
        if k % 4 == 0:
            full[:] = rng.random((16, 16)) < 0.9
        elif k % 4 == 1:
            full[rng.choice(16, 3, replace=False)] = True
        elif k % 4 == 2:
            full[:, rng.choice(16, 3, replace=False)] = True
        else:
            full[:] = rng.random((16, 16)) < 0.3
        r, c = np.nonzero(full)
        rows.append(16 * rb + r)
        cols.append(16 * cb + c)
    keys = wl.sorted_unique(np.concatenate(rows).astype(np.int64) * n + np.concatenate(cols))
    ptr, idx = wl.csr_from_sorted_keys(n, n, keys)
    return wl.CSR(n, n, ptr, idx, rng.choice(np.float32([1.5, -0.75, 0.125, 3.0, 0.0, -0.0, 2.0 ** -60, -2.0 ** -62]), keys.size).astype(np.float32))


@pytest.mark.parametrize("dtype", [B.F32, B.BF16, B.PATTERN])
@pytest.mark.parametrize("fmt", [B.FORMAT_AUTO, B.FORMAT_COO])
def test_payload_runs_once_per_four_columns(dtype, fmt):
    """x one entry short of, at and past the length from which payload runs are listed per four columns, from its list and from the
    masks, clustered and scattered, some entries twice; then a short x, to show that the staged x was cleared."""
    n = 160021
    csr = blocks_and_noise(n, 8)
    o = B.default_create_opts()
    o.force_format = fmt
    h = Handle(csr, dtype, opts=o)
    share = 1 - h.stats.class_nnz[B.BLK_INLINE] / h.stats.nnz
    assert 1 / 8 < share and (share < 1 / 2 or fmt == B.FORMAT_COO)          # (packed lists do not count towards the other half)
    A = ref_matrix(csr, bf16=dtype == B.BF16)
    P = oracle.RefMatrix(csr.m, csr.n, csr.row_ptr, csr.col_idx, None)
    rng = np.random.default_rng(1)
    runs = (np.arange(0, 24000, 3)[:, None] * 16 // 3 + np.arange(11)).ravel()            # 11 columns of every 16
    lists = [np.sort(rng.choice(n, k, replace=False)) for k in (8186, 8187)]               # 8191 and 8192 with the five twice
    lists += [runs[:9000], np.r_[runs[20000:29000], n - 1], runs[:40000], np.array([5, 700, n - 1])]
    for idx in lists:
        idx = idx.astype(np.int32)
        val = rng.choice(np.float32([1.0, -2.0, 0.5, -0.0, 2.0 ** -60]), idx.size).astype(np.float32)
        twice = rng.integers(0, idx.size, 5)                                             # (the same value: it contributes once)
        x = wl.SparseVec(n, idx, val)
        given = wl.SparseVec(n, np.r_[idx, idx[twice]], np.r_[val, val[twice]]) if idx.size > 256 else x
        for semiring in (B.OR_AND, B.MIN_PLUS) if dtype == B.PATTERN else (B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS):
            got = h.run(given, semiring=semiring)
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(P if dtype == B.PATTERN else A, x.idx, x.val)
                assert np.array_equal(got[0], wi) and np.array_equal(got[1], wv.astype(np.float32))
            else:
                check_against_oracle(got, oracle.ref_pull(P if dtype == B.PATTERN else A, x.idx, x.val), boolean=semiring == B.OR_AND)
            assert h.get_stats().last_path == B.PATH_PUSH
    h.close()


@pytest.mark.parametrize("m", [2048 * 1185, 2048 * 2400 + 7])               # two and three tiles per thread block
@pytest.mark.parametrize("dtype", [B.F32, B.PATTERN])
def test_wide_finish_with_private_accumulators(m, dtype):
    """The finishing kernel of several tiles per thread block behind a push that used private accumulators, with and without a row
    mask; an unrelated call afterwards shows that accumulators and private copies were left clear."""
    n = 40009
    csr = matrix(m, n, 5)
    h = Handle(csr, dtype)
    assert h.stats.n_hub_row_blocks > 0
    A = ref_matrix(csr) if dtype == B.F32 else None
    P = oracle.RefMatrix(csr.m, csr.n, csr.row_ptr, csr.col_idx, None)
    rng = np.random.default_rng(m)
    always = np.int32([3, 4, 21, 300, n - 1])
    hub_rows = np.bincount(np.repeat(np.arange(csr.m), np.diff(csr.row_ptr))[np.isin(csr.col_idx, always)], minlength=csr.m)
    drop = rng.random(m) < 0.5
    drop[33] = True                                                            # (the full row: its row block is a hub)
    drop[np.flatnonzero(hub_rows)[::3]] = True
    words = np.packbits(np.r_[drop, np.zeros(-m % 32, bool)], bitorder="little").view(np.int32)
    mask = torch.from_numpy(words.copy()).to("cuda")
    h.set_opts(no_small_call=1, hub_min_nnz_x=1)
    for k in (40, 600):                                                        # (at most n / 64 entries)
        idx = np.unique(np.r_[always, rng.choice(n, k - 5)]).astype(np.int32)
        x = wl.SparseVec(n, idx, rng.choice(np.float32([1.0, -2.0, 0.5, -0.0, 2.0 ** -60]), idx.size).astype(np.float32))
        xi, xv = torch.from_numpy(idx).to("cuda"), torch.from_numpy(x.val).to("cuda")
        for semiring in (B.OR_AND, B.MIN_PLUS) if dtype == B.PATTERN else (B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS):
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(P if dtype == B.PATTERN else A, x.idx, x.val)
                want = (wi, wv, np.abs(wv))
            else:
                want = oracle.ref_pull(P if dtype == B.PATTERN or semiring == B.OR_AND else A, x.idx, x.val)
            for complement in (None, 1, 0):
                if complement is None:
                    got, w = h.run(x, semiring=semiring), want
                else:
                    h.y_nnz.fill_(-7)
                    B.dbspmspv_run_masked(h.h, xi, xv, idx.size, semiring, mask, complement, h.y_idx, h.y_val, m, h.y_nnz)
                    kk = int(h.y_nnz.item())
                    got = (h.y_idx[:kk].cpu().numpy(), h.y_val[:kk].cpu().numpy(), kk)
                    keep = drop[want[0]] != bool(complement)
                    w = tuple(v[keep] for v in want)
                if semiring == B.MIN_PLUS:
                    assert np.array_equal(got[0], w[0]) and np.array_equal(got[1], w[1].astype(np.float32))
                else:
                    check_against_oracle(got, w, boolean=semiring == B.OR_AND)
            # an unrelated call, without private accumulators
            one = wl.SparseVec(n, np.int32([700]), np.float32([1.0]))
            h.set_opts(no_small_call=1, hub_min_nnz_x=-1)
            check_against_oracle(h.run(one, semiring=B.OR_AND), oracle.ref_pull(P, one.idx, one.val), boolean=True)
            h.set_opts(no_small_call=1, hub_min_nnz_x=1)
    h.close()


@pytest.mark.parametrize("tiles", [296, 297, 593, 1200])                     # one, two, three and four tiles per thread block (148 SMs)
def test_wide_finish_behind_a_push_of_whole_blocks(tiles):
    """A short x on a tall matrix whose elements sit in full blocks, rows at both ends of tiles among them, masked and not."""
    m, n = 2048 * tiles - 3, 40009
    rng = np.random.default_rng(tiles)
    rbs = np.unique(np.r_[0, 127, 128, m // 16 - 1, rng.integers(0, m // 16, 1500)])
    r = (16 * rbs[:, None] + np.arange(16)).reshape(-1, 16, 1)
    c = (16 * rng.integers(0, n // 16, rbs.size)[:, None] + np.arange(16)).reshape(-1, 1, 16)
    keys = wl.sorted_unique((r * np.int64(n) + c).ravel()[rng.random(rbs.size * 256) < 0.8])
    ptr, idx = wl.csr_from_sorted_keys(m, n, keys)
    csr = wl.CSR(m, n, ptr, idx, rng.choice(np.float32([1.5, -0.75, 0.0, -0.0, 2.0 ** -60]), keys.size).astype(np.float32))
    h, A = Handle(csr, B.F32), ref_matrix(csr)
    assert h.stats.class_nnz[B.BLK_INLINE] * 2 < h.stats.nnz
    drop = rng.random(m) < 0.5
    mask = torch.from_numpy(np.packbits(np.r_[drop, np.zeros(-m % 32, bool)], bitorder="little").view(np.int32).copy()).to("cuda")
    for k in (3, 312):                                                         # (at most n / 128 entries)
        at = np.unique(np.r_[csr.col_idx[:3], csr.col_idx[-3:], rng.choice(csr.col_idx, k)])[:312].astype(np.int32)
        x = wl.SparseVec(n, at, rng.choice(np.float32([1.0, -2.0, 2.0 ** -60]), at.size).astype(np.float32))
        xi, xv = torch.from_numpy(at).to("cuda"), torch.from_numpy(x.val).to("cuda")
        for semiring in (B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS):
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(A, x.idx, x.val)
                want = (wi, wv, np.abs(wv))
            else:
                want = oracle.ref_pull(A, x.idx, x.val)
            for complement in (None, 1):
                if complement is None:
                    got, w = h.run(x, semiring=semiring), want
                else:
                    B.dbspmspv_run_masked(h.h, xi, xv, at.size, semiring, mask, 1, h.y_idx, h.y_val, m, h.y_nnz)
                    kk = int(h.y_nnz.item())
                    got = (h.y_idx[:kk].cpu().numpy(), h.y_val[:kk].cpu().numpy(), kk)
                    w = tuple(v[~drop[want[0]]] for v in want)
                if semiring == B.MIN_PLUS:
                    assert np.array_equal(got[0], w[0]) and np.array_equal(got[1], w[1].astype(np.float32))
                else:
                    check_against_oracle(got, w, boolean=semiring == B.OR_AND)
    h.close()


# (148 SMs: more than one wave, one tile per thread block; from 1333 tiles on the handle of blocks takes pairs: a last pair of one tile, of two)
@pytest.mark.parametrize("m", [2048 * 1185 - 5, 2048 * 1186, 2048 * 1187 + 16, 2048 * 1333 - 5, 2048 * 1334, 2048 * 1335 + 16])
@pytest.mark.parametrize("blocks", [False, True])
def test_paired_finish(m, blocks):
    """The finishing kernel of two tiles per thread block behind a longer x, in turn with that of a short x on the same handle (another number of tiles per
    thread block); rows at both ends of tiles, full ones and empty ones, masked and not, a capacity in the middle of a tile."""
    n = 4001
    rng = np.random.default_rng(m)
    rows = np.unique(np.r_[0, 2047, 2048, 4095, 4096, m - 1, np.arange(6144, 10240), rng.integers(0, m, 40000)])
    if blocks:
        rbs = np.unique(rows // 16)[::4]
        rbs = rbs[rbs < m // 16]
        r = (16 * rbs[:, None] + np.arange(16)).reshape(-1, 16, 1)
        c = (16 * rng.integers(0, n // 16, rbs.size)[:, None] + np.arange(16)).reshape(-1, 1, 16)
        keys = wl.sorted_unique((r * np.int64(n) + c).ravel()[rng.random(rbs.size * 256) < 0.8])
    else:
        keys = wl.sorted_unique(np.r_[rows, rows].astype(np.int64) * n + rng.integers(0, n, 2 * rows.size))
    ptr, idx = wl.csr_from_sorted_keys(m, n, keys)
    csr = wl.CSR(m, n, ptr, idx, rng.choice(np.float32([1.5, -0.75, 0.0, -0.0, 2.0 ** -60]), keys.size).astype(np.float32))
    h, A = Handle(csr, B.F32), ref_matrix(csr)
    assert h.stats.n_hub_row_blocks == 0
    drop = rng.random(m) < 0.5
    mask = torch.from_numpy(np.packbits(np.r_[drop, np.zeros(-m % 32, bool)], bitorder="little").view(np.int32).copy()).to("cuda")
    h.set_opts(no_small_call=1)
    for k in (1500, 20, 200, 3900):
        at = rng.choice(n, k, replace=False).astype(np.int32)
        x = wl.SparseVec(n, at, rng.choice(np.float32([1.0, -2.0, 2.0 ** -60]), k).astype(np.float32))
        xi, xv = torch.from_numpy(at).to("cuda"), torch.from_numpy(x.val).to("cuda")
        for semiring in (B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS):
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(A, x.idx, x.val)
                want = (wi, wv, np.abs(wv))
            else:
                want = oracle.ref_pull(A, x.idx, x.val)
            got, w = h.run(x, semiring=semiring), want
            for masked in (False, True):
                if masked:
                    B.dbspmspv_run_masked(h.h, xi, xv, k, semiring, mask, 1, h.y_idx, h.y_val, m, h.y_nnz)
                    kk = int(h.y_nnz.item())
                    got = (h.y_idx[:kk].cpu().numpy(), h.y_val[:kk].cpu().numpy(), kk)
                    w = tuple(v[~drop[want[0]]] for v in want)
                if semiring == B.MIN_PLUS:
                    assert np.array_equal(got[0], w[0]) and np.array_equal(got[1], w[1].astype(np.float32))
                else:
                    check_against_oracle(got, w, boolean=semiring == B.OR_AND)
    cap = want[0].size // 3
    h.y_idx.fill_(-1)
    yi, _, kk = h.run(x, semiring=B.OR_AND, capacity=cap)
    assert kk == want[0].size and (h.y_idx[cap:].cpu().numpy() == -1).all()
    h.get_stats(raise_on_device_status=False)
    check_against_oracle(h.run(x, semiring=B.OR_AND), oracle.ref_pull(A, x.idx, x.val), boolean=True)
    h.close()
