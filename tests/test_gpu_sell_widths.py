"""Sliced-ELL PCG at the edges of the solver kernel's entry batches (eight entries of a row are
loaded together) and of its four-row and 32-row groups: rows of 1, 3, 7, 8, 9, 16, 17 and 40 entries,
few rows, several replacements and a stop in mid-solve, against the dense solution."""
import numpy as np
import pytest
import torch

from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu
sp = pytest.importorskip("scipy.sparse")


def band_spd(n, width, seed):
    """Symmetric, strictly diagonally dominant, rows of up to `width` entries on distant diagonals."""
    half = (width - 1) // 2
    A = sp.lil_matrix((n, n))
    off = [1 + (q * 37) % max(1, n - 1) for q in range(half)]
    for q, o in enumerate(sorted(set(off))):
        v = inputs.uniform_pm1(seed + q, 0, n, np.float64).astype(np.float32).astype(np.float64)
        for i in range(n - o):
            A[i, i + o] = A[i + o, i] = v[i]
    d = np.asarray(abs(A).sum(axis=1)).ravel()
    A.setdiag(np.float32(1.0) + d.astype(np.float32))
    A = A.tocsr()
    A.sort_indices()
    return A.astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("n,width", [(5, 3), (33, 1), (500, 7), (500, 8), (1000, 9), (97, 16), (1000, 17), (300, 40)])
def test_sell_pcg_row_widths(gpu_lib, n, width):
    A = band_spd(n, width, 70)
    b = inputs.uniform_pm1(71, 0, n, np.float64)
    m = gpu_lib.sell_from_csr(torch.from_numpy(A.indptr.astype(np.int64)).cuda(),
                              torch.from_numpy(A.indices.astype(np.int32)).cuda(),
                              torch.from_numpy(A.data.astype(np.float32)).cuda())
    bd = torch.from_numpy(b).cuda()
    x, res = gpu_lib.sell_pcg_solve(m, bd, tol=1e-10, maxit=2000)
    assert res["status"] == gpu_lib.OK, res
    xr = x.cpu().numpy()
    tr = np.linalg.norm(b - A @ xr) / np.linalg.norm(b)
    assert tr <= 1e-10 and abs(res["rel_res_true"] - tr) <= 1e-3 * tr + 1e-16
    # stopped after two iterations: x holds both updates (the reported residual is that of x)
    x2, r2 = gpu_lib.sell_pcg_solve(m, bd, tol=1e-14, maxit=2)
    t2 = np.linalg.norm(b - A @ x2.cpu().numpy()) / np.linalg.norm(b)
    assert abs(r2["rel_res_true"] - t2) <= 1e-3 * t2 + 1e-15
    assert t2 <= r2["rel_res_recursive"] * 1.001 + 1e-6
