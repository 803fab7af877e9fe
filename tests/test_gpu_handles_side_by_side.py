"""Handles of different sizes used in turn: what a call sets up for its kernels (shared-memory limits belong to the kernel, not
to the handle) holds for the other handles as well."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import Handle, DEV, TOL, check_against_oracle, ref_matrix

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("semiring", [B.PLUS_TIMES, B.OR_AND, B.MIN_PLUS, None], ids=["plus_times", "or_and", "min_plus", "decode"])
def test_pulls_on_a_large_a_small_and_the_large_handle(semiring):
    mats = [wl.random_sparse(3000, n, 4 * n, 7) for n in (1 << 20, 16384)]           # presence filters of 128 KB and 2 KB
    handles = [Handle(c, B.F32) for c in mats]
    for h in handles:
        h.set_opts(force_path=B.PATH_PULL)
    for h, c in [(handles[k], mats[k]) for k in (0, 1, 0, 1, 0)]:
        x = wl.sparse_x(3, 0, c.n, c.n // 2)
        A = ref_matrix(c)
        if semiring is None:
            xd = np.zeros(c.n, np.float32)
            xd[x.idx] = x.val
            y = torch.full((c.m,), 7.0, device=DEV)
            B.dbspmspv_decode(h.h, torch.from_numpy(xd).to(DEV), y)
            want, scale = oracle.ref_decode(A, xd)
            assert (np.abs(y.cpu().numpy() - want) <= TOL * scale).all()
        else:
            got = h.run(x, semiring=semiring)
            if semiring == B.MIN_PLUS:
                wi, wv = oracle.ref_minplus(A, x.idx, x.val)
                assert np.array_equal(got[0], wi) and np.array_equal(got[1], wv.astype(np.float32))
            else:
                check_against_oracle(got, oracle.ref_pull(A, x.idx, x.val), boolean=semiring == B.OR_AND)
        assert h.get_stats().last_path == B.PATH_PULL
    for h in handles:
        h.close()
