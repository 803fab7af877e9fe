"""From its second call on, a sequence of kernels is launched as a graph that the handle keeps, with
the arguments and grids of the new call; a call on a capturing stream becomes part of the
caller's graph instead.  Either way a call gives the oracle's result for its own x."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, DEV, check_against_oracle, ref_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(1, 40, 256), (300, 2000, 301), (5, 3000, 9000)], ids=["short", "general", "mixed"])
def test_repeated_calls_take_new_arguments(counts):
    csr = wl.rmat(14, 16, seed=6)
    A = ref_matrix(csr)
    h = Handle(csr, B.F32)
    streams = [torch.cuda.current_stream(), torch.cuda.Stream()]
    for rep in range(3):
        for i, k in enumerate(counts):
            x = wl.sparse_x(50 + 10 * rep + i, 0, csr.n, k)
            torch.cuda.synchronize()
            with torch.cuda.stream(streams[(rep + i) % 2]):
                check_against_oracle(h.run(x), oracle.ref_pull(A, x.idx, x.val))
    h.close()


@pytest.mark.parametrize("count", [64, 1500])
def test_calls_inside_a_captured_graph(count):
    csr = wl.rmat(13, 16, seed=8)
    A = ref_matrix(csr)
    h = Handle(csr, B.F32)
    x = wl.sparse_x(3, 0, csr.n, count)
    xi, xv = torch.from_numpy(x.idx).to(DEV), torch.from_numpy(x.val).to(DEV)

    def call():
        B.dbspmspv_run(h.h, xi, xv, count, B.PLUS_TIMES, h.y_idx, h.y_val, csr.m, h.y_nnz)

    call(); call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    want = oracle.ref_pull(A, x.idx, x.val)
    for scale in (1.0, -2.0):
        xv.copy_(torch.from_numpy((x.val * scale).astype(np.float32)))
        h.y_nnz.fill_(-7)
        g.replay()
        torch.cuda.synchronize()
        k = int(h.y_nnz.item())
        check_against_oracle((h.y_idx[:k].cpu().numpy(), h.y_val[:k].cpu().numpy(), k),
                             (want[0], want[1] * scale, want[2] * abs(scale)))
    check_against_oracle(h.run(x), want)                     # and ordinary calls afterwards
    h.close()


@pytest.mark.parametrize("where", ["same thread", "another thread"])
def test_calls_beside_a_capture(where):
    """While a stream is being captured in the global mode, calls on another stream that is not captured run as ever, and the
    capture goes on: first call, second (a graph is built), later ones."""
    import threading

    csr = wl.rmat(13, 16, seed=8)
    A = ref_matrix(csr)
    x = wl.sparse_x(3, 0, csr.n, 1500)
    want = oracle.ref_pull(A, x.idx, x.val)
    h = Handle(csr, B.F32)
    xi, xv = torch.from_numpy(x.idx).to(DEV), torch.from_numpy(x.val).to(DEV)
    side = torch.cuda.Stream()
    outs = [(torch.zeros(csr.m, dtype=torch.int32, device=DEV), torch.zeros(csr.m, device=DEV), torch.full((1,), -7, dtype=torch.int32, device=DEV)) for _ in range(4)]
    count = torch.zeros(4, device=DEV)
    errors = []

    def calls():
        try:
            for yi, yv, k in outs:
                B.dbspmspv_run(h.h, xi, xv, 1500, B.PLUS_TIMES, yi, yv, csr.m, k, side.cuda_stream)
                t = threading.Event()
                t.wait(0.05)                                  # (the stream is idle again: no call of the runtime may ask for it here)
        except Exception as e:                                # noqa: BLE001
            errors.append(e)

    count.add_(1.0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        count.add_(1.0)
        if where == "same thread":
            calls()
        else:
            t = threading.Thread(target=calls)
            t.start()
            t.join()
        count.mul_(2.0)
    assert not errors, errors
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert (count == 4.0).all()
    for yi, yv, k in outs:
        kk = int(k.item())
        check_against_oracle((yi[:kk].cpu().numpy(), yv[:kk].cpu().numpy(), kk), want)
    h.close()
