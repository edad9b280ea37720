"""Observables and integrated densities by two-part FP32 sums (fields of 2^15 points and
more, FP32 densities of any size) against the oracle: odd rows, several chunks and a
remainder per direction, planes, fields far from unit size (the observables' FP64 pass),
infinities and NaN.  Tolerance 1e-12 relative: a chain adds at most a few hundred terms
at 2^-48 each in two parts, eight in the densities', and the rest in FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1605_03958_gb300 as pkg
    return pkg


def make(P, orc, shape, prec, cplx, amp=1.0):
    p = orc.Problem(*shape, 0.3, 0.25, 0.4, 0.01, gamma=1.1, nu=1.7, lam=0.6, g=9.0)
    rng = np.random.default_rng(sum(shape))
    psi = amp * rng.standard_normal(p.shape)
    if cplx:
        psi = psi + 1j * amp * rng.standard_normal(p.shape)
    if prec == "f32":
        psi = psi.astype(np.complex64 if cplx else np.float32).astype(complex if cplx else float)
    s = P.Solver(*shape, 0.3, 0.25, 0.4, 0.01, 1.1, 1.7, 0.6, g=9.0, prec=prec)
    s.set_psi(psi)
    return p, s, psi


def check(orc, p, s, psi):
    o, r = s.observables(), orc.observables(p, psi)
    for k in r:
        if r[k] != 0:
            assert abs(o[k] - r[k]) <= TOL * abs(r[k]), (k, o[k], r[k])
    for a in range(3 if p.nz > 1 else 2):
        assert np.allclose(s.density1d(a), orc.density1d(p, psi, a), rtol=TOL, atol=0), a
    for a in range(3 if p.nz > 1 else 1):
        assert np.allclose(s.density2d(a), orc.density2d(p, psi, a), rtol=TOL, atol=0), a


@pytest.mark.parametrize("shape", [(65, 33, 17), (240, 70, 33), (1001, 40, 1), (3, 2048, 11), (2048, 9, 3), (35, 5, 203)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("cplx", [False, True])
def test_sums_match_oracle(P, orc, shape, prec, cplx):
    p, s, psi = make(P, orc, shape, prec, cplx)
    check(orc, p, s, psi)
    s.close()


@pytest.mark.parametrize("prec,amp", [("f32", 1e-12), ("f32", 1e15), ("f64", 1e-40), ("f64", 1e60)])
def test_fields_of_unusual_size(P, orc, prec, amp):
    p, s, psi = make(P, orc, (65, 33, 17), prec, True, amp)
    check(orc, p, s, psi)
    s.close()


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_bad_values_reach_every_sum_they_belong_to(P, orc, prec, bad):
    p, s, psi = make(P, orc, (65, 33, 17), prec, False)
    psi[5, 6, 7] = bad
    s.set_psi(psi)
    o = s.observables()
    assert not np.isfinite(o["norm"]) and not np.isfinite(o["energy"])
    for a, n in ((0, 7), (1, 6), (2, 5)):
        d = s.density1d(a)
        assert not np.isfinite(d[n]) and np.all(np.isfinite(np.delete(d, n)))
    assert not np.isfinite(s.density2d(0)[6, 7]) and not np.isfinite(s.density2d(1)[5, 7])
    s.close()
