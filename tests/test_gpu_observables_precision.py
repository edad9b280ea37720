"""Observables of fields of 2^15 points and more against sums in extended precision (numpy's long
double): smooth fields, coarsely and finely sampled.

Tolerance: FP64's.  The sums of threads, warps and blocks are added in FP64 by trees of about
twenty levels, each rounding 2^-53 of a partial sum at random signs, and a handful of products
follow: 8 x 2^-53 relative; the mean over several fields (no sum may lean to one side) 2 x 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
W = (1.1, 1.7, 0.6)


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1605_03958_gb300 as pkg
    return pkg


def exact(psi, h, g):
    Q = np.longdouble
    u = psi.astype(np.clongdouble if np.iscomplexobj(psi) else Q)
    sq = lambda v: v.real * v.real + (v.imag * v.imag if np.iscomplexobj(psi) else 0)
    nz, ny, nx = u.shape
    dV = Q(h) * Q(h) * (Q(h) if nz > 1 else 1)
    d = sq(u)
    x2, y2, z2 = (((np.arange(n) - Q(0.5) * (n - 1)) * Q(h)) ** 2 for n in (nx, ny, nz))
    sx, sy, sz = (d * x2[None, None, :]).sum(), (d * y2[None, :, None]).sum(), (d * z2[:, None, None]).sum()
    kin = Q(0)
    for ax in (2, 1) if nz == 1 else (2, 1, 0):
        kin += sq(np.diff(u, axis=ax)).sum() + sq(u.take(0, ax)).sum() + sq(u.take(-1, ax)).sum()
    o = dict(norm=d.sum() * dV, ekin=kin / (2 * Q(h) * Q(h)) * dV, eint=Q(g) / 2 * (d * d).sum() * dV,
             epot=(sx * Q(W[0]) ** 2 + sy * Q(W[1]) ** 2 + (sz * Q(W[2]) ** 2 if nz > 1 else 0)) / 2 * dV,
             rms_x=np.sqrt(sx / d.sum()), rms_y=np.sqrt(sy / d.sum()))
    if nz > 1:
        o["rms_z"] = np.sqrt(sz / d.sum())
    o["energy"] = o["ekin"] + o["epot"] + o["eint"]
    o["mu"] = o["energy"] + o["eint"]
    return o


@pytest.mark.parametrize("h", [0.02, 0.1])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(80, 70, 64), (45, 38, 34), (24, 40, 50), (600, 71, 1)])
def test_sums_are_fp64_sums(P, shape, cplx, prec, h):
    x, y, z = ((np.arange(n) - 0.5 * (n - 1)) * h for n in shape)
    off = {}
    for seed in range(4):
        f = 0.4 * np.exp(-0.4 * x * x)[None, None, :] * np.exp(-0.5 * y * y)[None, :, None] \
            * np.exp(-0.7 * z * z)[:, None, None] * (1 + 0.1 * np.cos(0.7 * x + 1.3 * seed))[None, None, :]
        if cplx:
            f = f * np.exp(0.4j * np.sin(x + 0.2 + seed))[None, None, :]
        if prec == "f32":
            f = f.astype(np.complex64 if cplx else np.float32).astype(f.dtype)
        s = P.Solver(*shape, h, dt=0.1 * h * h, gamma=W[0], nu=W[1], lam=W[2], g=9.0, prec=prec)
        s.set_psi(f)
        o = s.observables()
        s.close()
        for k, r in exact(f, h, 9.0).items():
            off.setdefault(k, []).append(float((o[k] - r) / r))
    for k, e in off.items():
        assert max(map(abs, e)) <= 8 * 2.0 ** -53, (k, e)
        assert abs(np.mean(e)) <= 2 * 2.0 ** -53, (k, e)
