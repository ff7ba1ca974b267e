"""Sliced-ELL PCG on matrices that are not positive definite: p.Ap <= 0 in the first iteration, in a
later one and at either side of a turn of the device-driven loop ends the solve with GBPCG_BREAKDOWN,
x holding the updates made before it.

Exact integers: blocks [[1, 2], [2, 1]] have the eigenvectors (1, 1) and (1, -1) for 3 and -1."""
import numpy as np
import pytest
import torch

from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu
sp = pytest.importorskip("scipy.sparse")


def dev(A):
    A = A.tocsr()
    A.sort_indices()
    return (torch.from_numpy(A.indptr.astype(np.int64)).cuda(), torch.from_numpy(A.indices.astype(np.int32)).cuda(),
            torch.from_numpy(A.data.astype(np.float32)).cuda())


def cg_until_breakdown(A, b, maxit):
    """Jacobi-PCG of a matrix with unit diagonal in FP64: (iterations, x) at p.Ap <= 0."""
    x, r = np.zeros_like(b), b.copy()
    p, rz = r.copy(), r @ r
    for it in range(maxit):
        q = A @ p
        if p @ q <= 0:
            return it, x
        a = rz / (p @ q)
        x = x + a * p
        r = r - a * q
        new = r @ r
        p = r + (new / rz) * p
        rz = new
    raise AssertionError("no breakdown")


@pytest.mark.parametrize("n", [2, 40, 1000])
def test_breakdown_in_the_first_iteration(gpu_lib, n):
    A = sp.block_diag([np.array([[1.0, 2.0], [2.0, 1.0]])] * (n // 2))
    m = gpu_lib.sell_from_csr(*dev(A))
    b = torch.from_numpy(np.tile([1.0, -1.0], n // 2)).cuda()
    x, res = gpu_lib.sell_pcg_solve(m, b, tol=1e-8, maxit=500)
    assert res["status"] == gpu_lib.BREAKDOWN and res["iters"] == 0, res
    assert not torch.any(x) and abs(res["rel_res_true"] - 1.0) <= 1e-12


def one_negative_eigenvalue(n):
    """Unit diagonal, eigenvalues between about 0.02 and 4 but one that is negative; entries exact in FP32."""
    Q, _ = np.linalg.qr(inputs.uniform_pm1(90, 0, n * n, np.float64).reshape(n, n))
    d = np.geomspace(0.02, 4.0, n)
    d[0] = -0.05
    A = (Q * d) @ Q.T
    t = 1.0 / np.sqrt(np.diag(A))
    A = (A * t[:, None] * t[None, :]).astype(np.float32).astype(np.float64)
    np.fill_diagonal(A, 1.0)
    return np.tril(A) + np.tril(A, -1).T


@pytest.mark.parametrize("weight", [1.0, 0.1, 1e-2, 1e-3])
def test_breakdown_in_a_later_iteration(gpu_lib, weight):
    """The less of the negative eigenvector b holds, the later p.Ap meets it (11, 19, 26 and 33 iterations;
    the loop takes eight a turn)."""
    n = 96
    A = one_negative_eigenvalue(n)
    lam, V = np.linalg.eigh(A)
    assert lam[0] < -1e-2 and lam[1] > 1e-2
    b = V[:, 1:] @ np.ones(n - 1) + weight * V[:, 0]
    it, _ = cg_until_breakdown(A, b, n)
    m = gpu_lib.sell_from_csr(*dev(sp.csr_matrix(A)))
    x, res = gpu_lib.sell_pcg_solve(m, torch.from_numpy(b).cuda(), tol=1e-13, maxit=10 * n)
    assert res["status"] == gpu_lib.BREAKDOWN, res
    assert abs(res["iters"] - it) <= 2, (res["iters"], it)
    true_rel = np.linalg.norm(b - A @ x.cpu().numpy()) / np.linalg.norm(b)
    assert abs(res["rel_res_true"] - true_rel) <= 1e-6 * true_rel
