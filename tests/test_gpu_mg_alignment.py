"""gbpcg_mg_vcycle on arrays that start at any element: the same bits as on aligned ones, for grids
whose level 0 runs in the vector kernels (constant and block coefficients, 4- and 2-wide rows below),
in the one-CTA tail and in the cluster sweeps; addresses inside an element are refused."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def rhs(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda") * 2 - 1


def at_offset(t, o):
    """A copy of t that starts o elements behind a 16-byte boundary."""
    buf = torch.empty(t.numel() + 8, dtype=t.dtype, device=t.device)
    assert buf.data_ptr() % 16 == 0
    v = buf[o:o + t.numel()].view(t.shape)
    v.copy_(t)
    return v


@pytest.mark.parametrize("shape,kb", [((32, 32, 32), None), ((64, 48, 40), 8), ((24, 40, 56), 5), ((16, 16, 16), None),
                                      ((31, 29, 36), None)])
def test_unaligned_vectors(gpu_lib, shape, kb):
    k = None
    if kb:
        k = torch.exp(rhs(tuple(-(-n // kb) for n in shape), 5))
    r = rhs(shape, 6)
    z, levels = gpu_lib.mg_vcycle(r, k_block=k, kb=kb or 8)
    for ro, zo in ((1, 0), (0, 1), (2, 3), (3, 2)):
        zu = at_offset(torch.zeros_like(z), zo)
        ru = at_offset(r, ro)
        out, lv = gpu_lib.mg_vcycle(ru, zu, k_block=k, kb=kb or 8)
        assert lv == levels and torch.equal(out, z) and torch.equal(ru, r), (ro, zo)


def test_addresses_inside_an_element_are_refused(gpu_lib):
    shape = (32, 32, 32)
    r = rhs(shape, 7)
    ws = gpu_lib.mg_workspace(shape)
    g = gpu_lib.make_grid(shape)
    buf = torch.empty(r.numel() + 8, device="cuda")
    for rp, zp in ((r.data_ptr() + 2, buf.data_ptr()), (r.data_ptr(), buf.data_ptr() + 1)):
        rc = gpu_lib.load().gbpcg_mg_vcycle(ctypes.byref(g), ctypes.c_void_p(rp), ctypes.c_void_p(zp),
                                            ctypes.c_void_p(ws.data_ptr()), ws.numel(), None, ctypes.c_void_p(0))
        assert rc == gpu_lib.ERR_ARG
