"""Which kernels a solve runs: the on-chip solver's three builds, one CTA, sums by slots (up to 32 CTAs)
and by inboxes (beyond), batches that share a launch, go one by one or stream, and grids that do not
fit.  The other tests of the on-chip solver compare results that the streaming passes would give too;
here the launches themselves are recorded by the profiler."""
import json

import pytest
import torch

from paper_2603_23343_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture
def launches(tmp_path):
    """launches(fn): [(kernel name, grid x)] of fn's solver kernels."""
    from torch.profiler import ProfilerActivity, profile

    def record(fn):
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            fn()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        events = json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
        return [(e["name"], e["args"]["grid"][0]) for e in events if e.get("cat") == "kernel"
                and any(k in e["name"] for k in ("resident_", "zmarch_kernel", "batch_kernel"))]

    def fn(f):
        f()  # the first call of a process may load kernels lazily
        k = record(f)
        return k if k else record(f)  # (the first trace of a process can come back empty)

    return fn


def rhs(shape, seed):
    return torch.from_numpy(inputs.uniform_rhs(shape, seed)).cuda()


@pytest.mark.parametrize("shape,build,ctas", [((8, 8, 8), 4, (1, 1)), ((1, 1, 9), 4, (1, 1)), ((32, 32, 32), 4, (2, 32)),
                                              ((61, 62, 63), 4, (33, 160)), ((64, 64, 64), 4, (33, 160)),
                                              ((128, 128, 128), 7, (33, 160)), ((64, 112, 512), 14, (33, 160)),
                                              ((160, 160, 160), 14, (33, 160))])
def test_a_grid_that_fits_takes_one_launch(gpu_lib, launches, shape, build, ctas):
    b = rhs(shape, 400)
    k = launches(lambda: gpu_lib.pcg_solve(b, tol=1e-3, maxit=5))
    assert len(k) == 1 and f"resident_kernel<512, {build}," in k[0][0], k
    assert ctas[0] <= k[0][1] <= ctas[1], k


def test_other_solves_take_the_passes(gpu_lib, launches):
    """A grid too large, rows too short, block coefficients, tiles asked for, 16-bit vectors."""
    code = gpu_lib.tile_cfg_code(0, 0)
    kb = torch.ones((4, 4, 4), device="cuda")
    b = rhs((32, 32, 32), 401)
    for f in (lambda: gpu_lib.pcg_solve(rhs((176, 176, 176), 402), tol=1e-3, maxit=3),
              lambda: gpu_lib.pcg_solve(rhs((9, 8, 7), 403), tol=1e-3, maxit=3),
              lambda: gpu_lib.pcg_solve(b, tol=1e-3, maxit=3, k_block=kb),
              lambda: gpu_lib.pcg_solve(b, tol=1e-3, maxit=3, tile_cfg=code),
              lambda: gpu_lib.pcg_solve(b.double(), tol=1e-3, maxit=3, storage=torch.float16)):
        k = launches(f)
        assert k and all("zmarch_kernel" in n for n, _ in k), k


def test_routes_of_a_batch(gpu_lib, launches):
    def names(shapes, **kw):
        bs = [rhs(s, 410 + i) for i, s in enumerate(shapes)]
        return [n for n, _ in launches(lambda: gpu_lib.pcg_solve_batched(bs, tol=1e-3, maxit=5, **kw))]

    def count(k, what):
        return sum(what in n for n in k)

    small, large, whole = (24, 20, 36), (120, 128, 128), (192, 192, 192)
    k = names([small] * 3 + [(17, 19, 23)])  # side by side
    assert len(k) == 1 and "resident_batch_kernel<256" in k[0], k
    k = names([small] * 3 + [large])  # the large one by itself
    assert len(k) == 2 and count(k, "resident_batch_kernel<256") == 1 and count(k, "resident_kernel<512") == 1, k
    k = names([whole, whole, small])  # what does not fit streams
    assert count(k, "resident") == 0 or count(k, "resident") < len(k), k
    k = names([small] * 3, tile_cfg=1)  # tiles asked for
    assert count(k, "resident") == 0, k
    k = names([small, (17, 19, 23), (64, 64, 64)], graph=True)  # the standalone solves' bricks, side by side
    assert k and all("resident_batch_kernel<512, 4" in n for n in k), k
