"""What a create needs beside its input: a matrix is built with little memory left, and an index that does not fit is left out."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2608_16308_b200 import binding as B
from paper_2608_16308_b200 import workloads as wl
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def test_index_by_weight_is_left_out_where_it_does_not_fit():
    """27-point operator on 102^3 cells (28 M elements, a good part of them in blocks).  With 100 bytes per stored element left every index is built; with 56 the
    runs by weight, whose sort is the peak of the build, do not fit, and the handle comes without them.  Weights of one: the distances are the
    Chebyshev distances on the grid, either way."""
    d = 102
    g = wl.stencil27(d, values=False)
    ptr, col = torch.from_numpy(g.row_ptr).to(DEV), torch.from_numpy(g.col_idx).to(DEV)
    val, dist = torch.ones(g.nnz, device=DEV), torch.empty(g.n, device=DEV)
    z, y, x = np.meshgrid(*[np.arange(d)] * 3, indexing="ij")
    want = np.maximum(np.maximum(abs(x - 50), abs(y - 3)), abs(z - 77)).reshape(-1)
    B.dbspmspv_destroy(B.dbspmspv_create_csr(g.m, g.n, g.nnz, ptr, col, val, B.F32))       # (the library's code is on the device)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    cudart, index = ctypes.CDLL("libcudart.so.12"), []
    for left in (100, 56):
        held = ctypes.c_void_p()
        assert cudart.cudaMalloc(ctypes.byref(held), ctypes.c_size_t(torch.cuda.mem_get_info()[0] - left * g.nnz)) == 0
        try:
            h = B.dbspmspv_create_csr(g.m, g.n, g.nnz, ptr, col, val, B.F32)
        finally:
            cudart.cudaFree(held)
        index.append(B.dbspmspv_get_stats(h).bfs_index_bytes)
        B.db_sssp(h, 50 + d * (3 + d * 77), dist)
        assert np.array_equal(dist.cpu().numpy(), want)
        B.dbspmspv_destroy(h)
    assert index[0] - index[1] == 8 * g.nnz + 4 * (2 * g.m + 1)
