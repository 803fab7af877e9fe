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
