"""Performance cases of the library: what its users have it do, over the sizes they do it at.

A case is a dict of plain values; ``kind`` names the path:

kernels   one step of a hand-written Krylov iteration from the three kernels: q = A p, p.q, r -= alpha q
pcg       one Jacobi-PCG solve (FP32 vectors, or 16-bit vectors with FP64 refinement)
batch     many independent Poisson solves in one call
mg        one PCG solve with the multigrid preconditioner
sell      one Jacobi-PCG solve of the assembled matrix in Sliced-ELL form
conv      one 3x3x3 convolution layer of the network: forward, data gradient, weight gradient
gradient  the network's weight gradient of one training pair: forward, loss, backward
fcg       one flexible-CG solve with the network as its preconditioner

``prepare`` makes the inputs, ``run`` is one pass through the public entry points, ``work`` the
bytes and operations the path cannot do without, ``exact`` the outputs in 64-bit plain torch.

Solutions of the FP64 entry points leave as float32: the solve's tolerance fixes no digit beyond
those.  The network's outputs and gradients leave as bfloat16, the precision of its activations.
"""
from __future__ import annotations

import math
import random

import torch
import torch.nn.functional as F

from paper_2603_23343_gb300 import binding as B
from paper_2603_23343_gb300 import learned

DTYPES = {"f32": torch.float32, "f64": torch.float64, "f16": torch.float16, "bf16": torch.bfloat16}
KB = 8  # edge of a coefficient block
BATCH_SIZES = (48, 64, 96, 128, 160)
# layers of the network whose three directions are all public, (input, output channels)
CONV_LAYERS = [(16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (48, 16), (16, 1)]
MACS_PER_VOXEL = 47088  # of the whole network, per voxel of the finest level


def listed():
    return [
        # the smallest calls: a user's own iteration on the smallest grid, launches and latency
        dict(name="kernels_32", kind="kernels", nx=32, ny=32, nz=32, dtype="f32", lognormal=False),
        # the same with a coefficient on a grid whose rows fit no alignment
        dict(name="kernels_odd", kind="kernels", nx=255, ny=187, nz=201, dtype="f32", lognormal=True),
        # the smallest solve (the paper's problem on 32^3, FP32 data)
        dict(name="pcg_32", kind="pcg", nx=32, ny=32, nz=32, io="f32", storage="f32", lognormal=False),
        # the grid of the paper's main table
        dict(name="pcg_paper", kind="pcg", nx=512, ny=112, nz=64, io="f64", storage="f32", lognormal=False),
        # the headline solve: 256^3 Poisson, FP64 b and x
        dict(name="pcg_256", kind="pcg", nx=256, ny=256, nz=256, io="f64", storage="f32", lognormal=False),
        # mixed precision on the lognormal operator, an uneven grid
        dict(name="pcg_mixed", kind="pcg", nx=224, ny=184, nz=200, io="f64", storage="f16", lognormal=True),
        # many grids of uneven size at once
        dict(name="batch_24", kind="batch", problems=24, shape_seed=2),
        # the fastest solver of the library on the lognormal operator
        dict(name="mg_256", kind="mg", nx=256, ny=256, nz=256, lognormal=True),
        # an assembled matrix with an odd number of rows
        dict(name="sell_odd", kind="sell", nx=117, ny=103, nz=91, lognormal=False),
        # the network's heaviest layer at the training size
        dict(name="conv_48_16", kind="conv", nx=128, ny=128, nz=128, ci=48, co=16),
        # one training pair at the training size
        dict(name="gradient_128", kind="gradient", nx=128, ny=128, nz=128),
        # a learned-preconditioner solve
        dict(name="fcg_64", kind="fcg", nx=64, ny=64, nz=64),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, step * round(v / step)))


def draw(rng: random.Random):
    kind = rng.choice(("kernels", "kernels", "pcg", "pcg", "pcg", "batch", "mg", "mg", "sell", "conv", "conv",
                       "gradient", "fcg"))
    if kind == "kernels":
        return dict(kind=kind, nx=_log_int(rng, 24, 288), ny=_log_int(rng, 24, 256), nz=_log_int(rng, 24, 224),
                    dtype=rng.choice(("f32", "f32", "bf16", "f16")), lognormal=rng.random() < 0.5)
    if kind == "pcg":
        storage = rng.choice(("f32", "f32", "f32", "f16", "bf16"))
        io = "f64" if storage != "f32" else rng.choice(("f32", "f64", "f64"))
        top = 96 if io == "f32" else 208  # FP32 x cannot hold 1e-6 on the finest grids
        step = rng.choice((1, 4, 8, 8))   # rows that TMA can and cannot take
        return dict(kind=kind, nx=_log_int(rng, 24, top, step), ny=_log_int(rng, 20, top), nz=_log_int(rng, 20, top),
                    io=io, storage=storage, lognormal=storage != "f32" or rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(3, 20), shape_seed=rng.randint(3, 10 ** 6))
    if kind == "mg":
        return dict(kind=kind, nx=_log_int(rng, 32, 256, 8), ny=_log_int(rng, 32, 256, 8),
                    nz=_log_int(rng, 32, 256, 8), lognormal=rng.random() < 0.5)
    if kind == "sell":
        return dict(kind=kind, nx=_log_int(rng, 20, 128), ny=_log_int(rng, 20, 112), nz=_log_int(rng, 20, 96),
                    lognormal=rng.random() < 0.5)
    if kind == "conv":
        ci, co = rng.choice(CONV_LAYERS)
        return dict(kind=kind, nx=rng.choice((32, 64, 128)), ny=rng.choice((32, 64, 128)),
                    nz=rng.choice((32, 64, 128)), ci=ci, co=co)
    if kind == "gradient":
        return dict(kind=kind, nx=rng.choice((32, 64, 128)), ny=rng.choice((32, 64, 128)),
                    nz=rng.choice((32, 64, 128)))
    return dict(kind=kind, nx=rng.choice((32, 64)), ny=rng.choice((32, 64)), nz=rng.choice((32, 64)))


# ------------------------------------------------------------------ inputs --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(shape, g, dtype=torch.float32):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype) * 2 - 1


def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _coefficient(c, g):
    """Lognormal coefficient per 8^3 block, or None."""
    if not c.get("lognormal", False):
        return None
    nb = tuple(-(-n // KB) for n in _shape(c))
    return torch.exp(torch.randn(nb, generator=g, device="cuda"))


def _batch_shapes(c):
    rng = random.Random(c["shape_seed"])
    return [tuple(rng.choice(BATCH_SIZES) for _ in range(3)) for _ in range(c["problems"])]


def _network_weights(g, passing=False):
    """He-normal weights; `passing`: weights that pass the scaled residual through, slightly perturbed,
    so that the solve they precondition converges whatever the seed."""
    parts = []
    for name, ci, co in B.NN_LAYERS:
        std = math.sqrt(2.0 / (27 * ci)) * (0.5 if name == "c9" else 1.0)
        parts.append(torch.randn(co * 27 * ci, generator=g, device="cuda") * std)
    w = torch.cat(parts)
    return learned.identity_weights().cuda() + 0.02 * w if passing else w


def prepare(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    if kind == "batch":
        bs = [_uniform(s, g) for s in _batch_shapes(c)]
        xs = [torch.zeros_like(b) for b in bs]
        return dict(kind=kind, bs=bs, xs=xs, ws=_batch_workspace(bs))
    shape = _shape(c)
    if kind == "kernels":
        t = DTYPES[c["dtype"]]
        k = _coefficient(c, g)
        p, r = _uniform(shape, g).to(t), _uniform(shape, g).to(t)
        return dict(kind=kind, p=p, r=r, q=torch.empty_like(p), k=k, alpha=_alpha(c),
                    pq=torch.empty((), dtype=torch.float64, device="cuda"),
                    ws=torch.empty(B.dot_workspace_size(), dtype=torch.uint8, device="cuda"))
    if kind == "pcg":
        k = _coefficient(c, g)
        b = _uniform(shape, g).to(DTYPES[c["io"]])
        st, io = B._DTYPES[DTYPES[c["storage"]]], B._DTYPES[DTYPES[c["io"]]]
        return dict(kind=kind, b=b, x=torch.zeros_like(b), k=k, tol=_tol(c),
                    storage=None if c["storage"] == "f32" else DTYPES[c["storage"]],
                    ws=B.alloc_workspace(shape, k, KB, io_dtype=io, storage=st))
    if kind == "mg":
        k = _coefficient(c, g)
        b = _uniform(shape, g).double()
        return dict(kind=kind, b=b, x=torch.zeros_like(b), k=k, ws=B.mg_workspace(shape, k, KB))
    if kind == "sell":
        k = _coefficient(c, g)
        b = _uniform(shape, g).double().reshape(-1)
        return dict(kind=kind, m=B.sell_from_stencil(shape, k, KB), b=b, x=torch.zeros_like(b))
    if kind == "conv":
        x, w, gy = _layer(c, g)
        return dict(kind=kind, x=x, w=w, gy=gy, ws=B.conv3_workspace(shape, c["ci"], c["co"]))
    if kind == "gradient":
        k, r, e, w = _pair(c, g)
        return dict(kind=kind, k=k, r=r, e=e, w=w, ws=B.nn_workspace(shape, True))
    w = _network_weights(g, passing=True)
    k = _coefficient(dict(c, lognormal=True), g)
    b = _uniform(shape, g).double()
    return dict(kind=kind, w=w, k=k, b=b, x=torch.zeros_like(b), ws=B.fcg_workspace(shape, k, KB))


def _alpha(c):
    return 1.0 / sum(2.0 * (n + 1) ** 2 for n in _shape(c))


def _tol(c):
    return 1e-6 if c.get("storage", "f32") == "f32" else 1e-8


def _batch_workspace(bs):
    import ctypes
    n = len(bs)
    grids = (B.Grid * n)(*[B.make_grid(b.shape) for b in bs])
    o = B.make_opts(tol=1e-6, maxit=5000, io_dtype=B._DTYPES[bs[0].dtype])
    nbytes = ctypes.c_size_t(0)
    if B.load().gbpcg_workspace_size_batched(n, grids, ctypes.byref(o), ctypes.byref(nbytes)) != B.OK:
        raise RuntimeError(B.last_error())
    return torch.empty(nbytes.value, dtype=torch.uint8, device="cuda")


def _layer(c, g):
    """Activations after a ReLU, He-normal weights and an output gradient of one layer, BF16."""
    shape, ci, co = _shape(c), c["ci"], c["co"]
    x = F.relu(torch.randn((*shape, ci), generator=g, device="cuda")).bfloat16()
    w = (torch.randn((co, 27, ci), generator=g, device="cuda") * math.sqrt(2.0 / (27 * ci))).bfloat16()
    gy = (torch.randn((*shape, co), generator=g, device="cuda") * 0.1).bfloat16()
    return x, w, gy


def _pair(c, g):
    """A training pair (r = A e, e) on the lognormal operator, e a smooth error field of unit scale."""
    shape = _shape(c)
    k = _coefficient(dict(c, lognormal=True), g)
    e = _poisson_solve(_uniform(shape, g, torch.float64))
    e = e / e.square().mean().sqrt()
    e = (e + 0.02 * _uniform(shape, g, torch.float64)).float()
    r = _apply(e.double(), k).float()
    return k, r, e, _network_weights(g)


# -------------------------------------------------------------------- pass --

def run(s):
    kind = s["kind"]
    if kind == "kernels":
        q = B.stencil_apply(s["p"], s["q"], k_block=s["k"], kb=KB)
        pq = B.dot(s["p"], q, s["pq"], s["ws"])
        r = B.axpy(-s["alpha"], q, s["r"])
        return {"q": q, "pq": pq, "r": r}
    if kind == "pcg":
        s["x"].zero_()
        x, res = B.pcg_solve(s["b"], s["x"], tol=s["tol"], maxit=5000, k_block=s["k"], kb=KB, workspace=s["ws"],
                             storage=s["storage"])
        return {"x": x.float(), "status": res["status"]}
    if kind == "batch":
        torch._foreach_zero_(s["xs"])
        xs, res = B.pcg_solve_batched(s["bs"], s["xs"], tol=1e-6, maxit=5000, workspace=s["ws"])
        return {"x": xs, "status": [r["status"] for r in res]}
    if kind == "mg":
        s["x"].zero_()
        x, res = B.mg_pcg_solve(s["b"], s["x"], tol=1e-6, maxit=500, k_block=s["k"], kb=KB, workspace=s["ws"])
        return {"x": x.float(), "status": res["status"]}
    if kind == "sell":
        s["x"].zero_()
        x, res = B.sell_pcg_solve(s["m"], s["b"], s["x"], tol=1e-6, maxit=5000)
        return {"x": x.float(), "status": res["status"]}
    if kind == "conv":
        y = B.conv3_forward(s["x"], s["w"], workspace=s["ws"])
        gx = B.conv3_backward_data(s["gy"], s["w"], workspace=s["ws"])
        gw = B.conv3_backward_weight(s["x"], s["gy"], workspace=s["ws"])
        return {"y": y, "gx": gx, "gw": gw}
    if kind == "gradient":
        z = B.nn_forward(s["w"], s["r"], k_block=s["k"], kb=KB, workspace=s["ws"])
        _, gz = B.nn_loss(z, s["e"], s["ws"], k_block=s["k"], kb=KB)
        gw = B.nn_backward(gz, s["ws"], k_block=s["k"], kb=KB)
        return {"z": z.bfloat16(), "gz": gz.bfloat16(), "gw": gw.bfloat16()}
    s["x"].zero_()
    x, res = B.fcg_solve(s["w"], s["b"], s["x"], tol=1e-6, maxit=3000, k_block=s["k"], kb=KB, workspace=s["ws"])
    return {"x": x.float(), "status": res["status"]}


# -------------------------------------------------------------------- work --

def _iterations(shape, tol, lognormal):
    """Jacobi-PCG iterations from the spectrum of the operator: half the square root of its condition
    number times ln(2 / tol), of which a uniform right-hand side takes 0.57 (a lognormal coefficient
    about a fifth more)."""
    cond = 4 * sum((n + 1) ** 2 for n in shape) / (3 * math.pi ** 2)
    return max(1.0, 0.57 * 0.5 * math.sqrt(cond) * math.log(2 / tol) * (1.2 if lognormal else 1.0))


def work(c):
    kind = c["kind"]
    if kind == "batch":
        pts = [(s, math.prod(s)) for s in _batch_shapes(c)]
        return {"bytes": sum(8 * n for _, n in pts),
                "flops": sum(25.0 * n * _iterations(s, 1e-6, False) for s, n in pts)}
    shape = _shape(c)
    n = math.prod(shape)
    if kind == "kernels":  # reads p and r, writes q and r
        e = {"f32": 4, "f16": 2, "bf16": 2}[c["dtype"]]
        return {"bytes": 4 * e * n, "flops": 13.0 * n}
    if kind == "pcg":  # reads b, writes x
        return {"bytes": (8 if c["io"] == "f32" else 16) * n,
                "flops": 25.0 * n * _iterations(shape, _tol(c), c["lognormal"])}
    if kind == "mg":  # about 27 iterations of a solver step and a V-cycle
        return {"bytes": 16 * n, "flops": 27 * 75.0 * n}
    if kind == "sell":  # reads the matrix (7 entries of 8 bytes a row) and b, writes x
        return {"bytes": 76 * n, "flops": 25.0 * n * _iterations(shape, 1e-6, c["lognormal"])}
    if kind == "conv":
        ci, co = c["ci"], c["co"]
        return {"bytes": n * (2 * ci + 4 * co + 2 * co + 4 * ci), "flops": 3 * 2.0 * 27 * ci * co * n}
    if kind == "gradient":  # reads r and e, writes z and gz; forward and two backward products
        return {"bytes": 16 * n, "flops": 3 * 2.0 * MACS_PER_VOXEL * n}
    return {"bytes": 16 * n, "flops": 2.0 * MACS_PER_VOXEL * n * _iterations(shape, 1e-6, True)}


# ------------------------------------------------------- values in 64 bits --

def _field(k, shape):
    for d in range(3):
        k = k.repeat_interleave(KB, d)
    return k[:shape[0], :shape[1], :shape[2]].double()


def _faces(k, shape):
    """Per axis the n + 1 face coefficients over h^2: harmonic means, the cell's own value outside."""
    faces = []
    for d, n in enumerate(shape):
        s = float(n + 1) ** 2
        if k is None:
            faces.append(s)
            continue
        lo, hi = k.narrow(d, 0, n - 1), k.narrow(d, 1, n - 1)
        faces.append(torch.cat([k.narrow(d, 0, 1), 2 * lo * hi / (lo + hi), k.narrow(d, n - 1, 1)], d) * s)
    return faces


def _apply(u, k, faces=None):
    faces = _faces(None if k is None else _field(k, u.shape), u.shape) if faces is None else faces
    out = torch.zeros_like(u)
    for d, n in enumerate(u.shape):
        edge = torch.zeros_like(u.narrow(d, 0, 1))
        flux = torch.diff(torch.cat([edge, u, edge], d), dim=d) * faces[d]
        out -= torch.diff(flux, dim=d)
    return out


def _poisson_solve(b):
    """The solution of the constant-coefficient problem, by its sine eigenvectors."""
    x, lam = b.double(), 0.0
    bases = []
    for d, n in enumerate(b.shape):
        i = torch.arange(1, n + 1, dtype=torch.float64, device=b.device)
        bases.append(torch.sin(math.pi / (n + 1) * torch.outer(i, i)) * math.sqrt(2.0 / (n + 1)))
        lam = lam + (4.0 * (n + 1) ** 2 * torch.sin(math.pi * i / (2 * (n + 1))) ** 2).reshape(
            [-1 if a == d else 1 for a in range(3)])

    def both(x):
        x = torch.einsum("ai,ijk->ajk", bases[0], x)
        x = torch.einsum("bj,ajk->abk", bases[1], x)
        return torch.einsum("ck,abk->abc", bases[2], x)
    return both(both(x) / lam)


def _solve(b, k):
    if k is None:
        return _poisson_solve(b)
    b = b.double()
    faces = _faces(_field(k, b.shape), b.shape)
    diag = sum(f.narrow(d, 0, n) + f.narrow(d, 1, n) for (d, n), f in zip(enumerate(b.shape), faces))
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag
    p, rz, stop = z.clone(), torch.dot(r.flatten(), z.flatten()), 1e-12 * float(b.norm())
    for i in range(6000):
        q = _apply(p, None, faces)
        a = rz / torch.dot(p.flatten(), q.flatten())
        x += a * p
        r -= a * q
        if i % 16 == 15 and float(r.norm()) <= stop:
            break
        z = r / diag
        new = torch.dot(r.flatten(), z.flatten())
        p = z + (new / rz) * p
        rz = new
    return x


def _conv(x, w):
    """3x3x3 convolution, channels last, zero padding; w (co, 27, ci), tap (dz + 1) * 9 + (dy + 1) * 3 + dx + 1."""
    nz, ny, nx, _ = x.shape
    xp = F.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    y = 0
    for t in range(27):
        a, b, c = t // 9, t // 3 % 3, t % 3
        y = y + xp[a:a + nz, b:b + ny, c:c + nx] @ w[:, t].T
    return y


def _network(w, r, k):
    """z = N(r) of the U-net, the scale rms(D^{-1/2} r) a constant of the gradient."""
    ws, o = {}, 0
    for name, ci, co in B.NN_LAYERS:
        ws[name] = w[o:o + co * 27 * ci].reshape(co, 27, ci)
        o += co * 27 * ci
    kf = _field(k, r.shape)
    diag = sum(f.narrow(d, 0, n) + f.narrow(d, 1, n) for (d, n), f in zip(enumerate(r.shape), _faces(kf, r.shape)))
    s = r / diag.sqrt()
    rms = s.square().mean().sqrt()

    def pool(a):
        return F.avg_pool3d(a.permute(3, 0, 1, 2), 2).permute(1, 2, 3, 0)

    def up(a):
        return a.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)

    e0 = F.relu(_conv(F.relu(_conv(torch.stack([s / rms, kf.log()], 3), ws["c1"])), ws["c2"]))
    e1 = F.relu(_conv(F.relu(_conv(pool(e0), ws["c3"])), ws["c4"]))
    a6 = F.relu(_conv(F.relu(_conv(pool(e1), ws["c5"])), ws["c6"]))
    a7 = F.relu(_conv(torch.cat([up(a6), e1], 3), ws["c7"]))
    a8 = F.relu(_conv(torch.cat([up(a7), e0], 3), ws["c8"]))
    return rms * _conv(a8, ws["c9"])[..., 0] / diag.sqrt()


def exact(case, seed):
    c, g, kind = case, _gen(seed), case["kind"]
    if kind == "batch":
        return {"x": [_poisson_solve(_uniform(s, g)) for s in _batch_shapes(c)], "status": [None] * c["problems"]}
    shape = _shape(c)
    if kind == "kernels":
        t = DTYPES[c["dtype"]]
        k = _coefficient(c, g)
        p, r = _uniform(shape, g).to(t).double(), _uniform(shape, g).to(t).double()
        q = _apply(p, k)
        return {"q": q, "pq": (p * q).sum(), "r": r - _alpha(c) * q}
    if kind in ("pcg", "mg", "sell"):
        k = _coefficient(c, g)
        x = _solve(_uniform(shape, g), k)
        return {"x": x.reshape(-1) if kind == "sell" else x, "status": None}
    if kind == "conv":
        x, w, gy = _layer(c, g)
        x, w = x.double().requires_grad_(), w.double().requires_grad_()
        y = _conv(x, w)
        gx, gw = torch.autograd.grad(y, (x, w), gy.double())
        return {"y": y, "gx": gx, "gw": gw}
    if kind == "gradient":
        k, r, e, w = _pair(c, g)
        w = w.double().requires_grad_()
        e = e.double()
        z = _network(w, r.double(), k)
        zl = z.detach().requires_grad_()
        ae = _apply(e, k)
        a, cc, ee = (zl * ae).sum(), (zl * _apply(zl, k)).sum(), (e * ae).sum()
        gz, = torch.autograd.grad(0.5 * (1 - a * a.abs() / (cc * ee)), zl)
        gw, = torch.autograd.grad(z, w, gz)
        return {"z": z, "gz": gz, "gw": gw}
    _network_weights(g, passing=True)
    k = _coefficient(dict(c, lognormal=True), g)
    return {"x": _solve(_uniform(shape, g), k), "status": None}
