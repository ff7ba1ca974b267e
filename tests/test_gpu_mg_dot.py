"""r.z of the multigrid-preconditioned solver, summed in the V-cycle's last kernel, against the FP64 dot
product of the same vectors, on a grid where a thread sums about two hundred terms: one large term and
many that are each below half an ulp of it (a plain FP32 sum per thread: 6e-8 to 9e-8 off).

A solve stopped after one iteration leaves the start's r.z in its state, the first double of the
workspace (r = b for x0 = 0; the V-cycle after the last iteration is not run).  Bound: each thread's
compensated sum is good to its rounding to FP32, five FP32 additions across a warp follow, FP64 beyond.
Six roundings of at most 2^-24, independent in the 16,000 threads or more that hold large terms: 1e-9 of
the sum of |r z| in the mean square; ten times that."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kb", [None, 8, 5])
@pytest.mark.parametrize("every", [54, 53])
def test_rz_of_a_large_grid(gpu_lib, kb, every):
    n = 256
    g = torch.Generator(device="cuda").manual_seed(12)
    k = torch.exp(0.5 * torch.randn((-(-n // kb),) * 3, generator=g, device="cuda")) if kb else None
    b = torch.ones((n, n, n), dtype=torch.float64, device="cuda")
    b[::every] = 2.0 ** 19  # (max |b| below 2^20: the solve does not scale it)
    z, _ = gpu_lib.mg_vcycle(b.float(), k_block=k, kb=kb or 8)
    ws = gpu_lib.mg_workspace((n, n, n), k, kb or 8)
    _, res = gpu_lib.mg_pcg_solve(b, tol=1e-12, maxit=1, k_block=k, kb=kb or 8, workspace=ws)
    assert res["iters"] == 1 and res["status"] == gpu_lib.NOT_CONVERGED
    rz = float(ws[:8].view(torch.float64))
    terms = b * z.double()
    assert abs(rz - float(terms.sum())) <= 1e-8 * float(terms.abs().sum())
