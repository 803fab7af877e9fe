"""The decode over columns of bf16 layers (automatic mode, 1024 rows or more): strips of 64 rows, one or
several thread blocks per strip, one to nine vectors, sizes off every tile edge, activation options,
non-finite activations, a weight that is stored as -0."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, ref_matrix, DEV, TOL

pytestmark = pytest.mark.gpu


def bits(a):
    return torch.from_numpy(wl.f32_to_bf16_bits(a).view(np.int16)).to(DEV)


def check(y, want, scale):
    fin = np.isfinite(want)
    assert (np.isnan(y) == np.isnan(want)).all() and (y[np.isinf(want)] == want[np.isinf(want)]).all()
    assert (np.abs(y[fin].astype(np.float64) - want[fin]) <= TOL * scale[fin]).all()
    assert (y[fin & (scale == 0)] == 0.0).all()


# 17 / 18 strips (8 blocks each), 38 (2), 75 (1), 16 (8); rows and columns off the tiles, and a wide one
@pytest.mark.parametrize("shape,prune", [((1025, 333), 0.5), ((1100, 1000), 0.7), ((2400, 17), 0.6), ((4768, 260), 0.5), ((1024, 12289), 0.5)])
@pytest.mark.parametrize("x_f32", [0, 1])
def test_decode_over_columns(shape, prune, x_f32):
    m, n = shape
    w = wl.pruned_weight(m, n, prune, seed=5, stream=m + n)
    w.val[3] = np.float32(-0.0)
    h = Handle(w, B.BF16)
    A = ref_matrix(w, bf16=True)
    nv, ldx, ldy = 9, n + (8 if n % 8 == 0 else 3), m + 5
    xs = np.zeros((nv, ldx), np.float32)
    for b, zf in enumerate((0.7, 0.9, 0.05, 1.0, 0.99, 0.3, 0.8, 0.6, 0.95)):
        if zf < 1.0:
            xs[b, :n] = wl.relu_activation(n, zf, seed=5, stream=90 + b)
    xs[2, :n] *= np.where(np.arange(n) % 3 == 0, -1.0, 1.0)
    for special in (False, True):
        if special:
            xs[1, w.col_idx[5]], xs[1, w.col_idx[-1]] = np.inf, np.nan
        xr = wl.bf16_bits_to_f32(wl.f32_to_bf16_bits(xs))
        xd = torch.from_numpy(xs * np.float32(1 + 2.0 ** -11)).to(DEV) if x_f32 else bits(xs)      # (rounds back to the bf16 values)
        for relu, tau in ((0, 0.0), (1, 0.3)):
            h.set_opts(decode_relu=relu, decode_threshold=tau, decode_x_f32=x_f32)
            refs = []
            for b in range(nv):
                xt = xr[b, :n]
                with np.errstate(invalid="ignore"):
                    keep = ~(xt <= np.float32(tau)) if relu else ~(np.abs(xt) <= np.float32(tau))
                refs.append(oracle.ref_decode(A, np.where(keep, xt, 0.0).astype(np.float32)) + (keep,))
            for batch in (1, 2, 4, 5, 9):
                y = torch.full((batch, ldy), 55.0, device=DEV)
                before = h.get_stats().kernel_launches
                if batch == 1:
                    B.dbspmspv_decode(h.h, xd, y)
                    torch.cuda.synchronize()
                    assert h.get_stats().kernel_launches - before == 1
                    pad = np.zeros((n + 15) // 16 * 16, bool)
                    pad[:n] = refs[0][2]
                    assert h.get_stats().last_n_nzblk == int(pad.reshape(-1, 16).any(axis=1).sum())
                else:
                    B.dbspmspv_decode_batch(h.h, xd, ldx, y, ldy, batch)
                torch.cuda.synchronize()
                yh = y.cpu().numpy()
                for b in range(batch):
                    check(yh[b, :m], *refs[b][:2])
                assert (yh[:, m:] == 55.0).all()
    h.close()


def check_batches_in_a_row(m, n, launches):
    """Batches without any active entry, with a non-finite one and ordinary ones, one behind the other on one stream into one y
    that held NaN: every result is complete, whatever way the kernels of the call before it left."""
    w = wl.pruned_weight(m, n, 0.5, seed=11, stream=m)
    h = Handle(w, B.BF16)
    A = ref_matrix(w, bf16=True)
    nv = 8
    kinds = {"zero": np.zeros((nv, n), np.float32), "plain": np.stack([wl.relu_activation(n, 0.7, seed=11, stream=b) for b in range(nv)])}
    kinds["inf"] = kinds["plain"][::-1].copy()
    kinds["inf"][5, w.col_idx[7]] = np.inf
    refs = {k: [oracle.ref_decode(A, wl.bf16_bits_to_f32(wl.f32_to_bf16_bits(v[b])))[:2] for b in range(nv)] for k, v in kinds.items()}
    dev = {k: bits(v) for k, v in kinds.items()}
    y = torch.full((nv, m), float("nan"), device=DEV)
    order = ["zero", "plain", "inf", "zero", "inf", "plain", "zero", "zero", "inf", "inf", "plain", "plain"] * 4
    before, got = h.get_stats().kernel_launches, []
    for k in order:
        B.dbspmspv_decode_batch(h.h, dev[k], n, y, m, nv)
        got.append((k, y.clone()))
    torch.cuda.synchronize()
    assert h.get_stats().kernel_launches - before == launches * len(order)
    for k, t in got:
        th = t.cpu().numpy()
        for b in range(nv):
            check(th[b], *refs[k][b])
    h.close()


def test_batches_in_a_row_over_columns():
    check_batches_in_a_row(2400, 1040, 2)


def test_batches_in_a_row_over_blocks():
    check_batches_in_a_row(1008, 1040, 4)           # (too few rows for the column copy: tensor-core kernel and its two fallbacks)


# one thread block per strip: up to 8192 columns are a warp's first round over x, the widest layer fills the lists' shared memory exactly; two per strip: up to 16384
@pytest.mark.parametrize("shape", [(4768, 8191), (4768, 8192), (4768, 8193), (4800, 10000), (4768, 25600), (4000, 16385), (4000, 25600)])
def test_one_vector_of_more_than_one_round(shape):
    """Single vectors whose warps take more than one round over x: every entry active, a third of them scattered, in runs, only columns of the later rounds, and a
    non-finite entry in the first, in a later round and in both."""
    m, n = shape
    gen = torch.Generator(device=DEV).manual_seed(n)
    keep = torch.rand((m, n), generator=gen, device=DEV) < 0.3
    val = torch.randn((m, n), generator=gen, device=DEV).to(torch.bfloat16).float()
    val[val == 0] = 0.5
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(keep.sum(dim=1), 0, out=ptr[1:])
    w = wl.CSR(m, n, ptr.cpu().numpy(), keep.nonzero()[:, 1].to(torch.int32).cpu().numpy(), val[keep].cpu().numpy())
    del val
    h, A = Handle(w, B.BF16), ref_matrix(w, bf16=True)
    rng = np.random.default_rng(m + n)
    full = np.where(rng.random(n) < 0.5, -1.0, 1.0) * (0.1 + rng.random(n))
    cut = 16384 if m < 4737 else 8192
    late = np.arange(n) >= min(cut, n - 16)
    runs = (np.arange(n) // 192) % 3 == 1
    xs = [full, full * (rng.random(n) < 0.3), full * runs, full * late, full * (rng.random(n) < 0.1)]
    for at in ([5], [n - 3], [7, n - 1]):
        xs.append(full * (rng.random(n) < 0.3))
        xs[-1][at] = np.array([np.inf, np.nan][:len(at)])
    for x in xs:
        x = wl.bf16_bits_to_f32(wl.f32_to_bf16_bits(x.astype(np.float32)))
        y = torch.full((m + 3,), 55.0, device=DEV)
        before = h.get_stats().kernel_launches
        B.dbspmspv_decode(h.h, bits(x), y)
        torch.cuda.synchronize()
        st = h.get_stats()
        assert st.kernel_launches - before == 1
        active = np.zeros((n + 15) // 16 * 16, bool)
        active[:n] = x != 0
        assert st.last_n_nzblk == int(active.reshape(-1, 16).any(axis=1).sum())
        yh = y.cpu().numpy()
        check(yh[:m], *oracle.ref_decode(A, x)[:2])
        assert (yh[m:] == 55.0).all()
    h.close()
