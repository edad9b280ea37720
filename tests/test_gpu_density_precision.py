"""Integrated densities of FP32 fields against sums in extended precision (numpy's long double).

Tolerance: FP64's.  A density is a sum of at most 2^11 terms per line in FP64 (rounding errors of
2^-53 of the partial sums at random signs, a few times 2^-53 in all); what is summed in FP32
arithmetic first must not show: 8 x 2^-53 relative for every value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1605_03958_gb300 as pkg
    return pkg


H = (0.3, 0.25, 0.4)


def exact(psi):
    d = psi.real.astype(np.longdouble) ** 2 + psi.imag.astype(np.longdouble) ** 2
    hx, hy, hz = (np.longdouble(h) for h in H)
    hz = hz if psi.shape[0] > 1 else np.longdouble(1)
    return ([d.sum((0, 1)) * hy * hz, d.sum((0, 2)) * hx * hz, d.sum((1, 2)) * hx * hy],
            [d.sum(0) * hz, d.sum(1) * hy, d.sum(2) * hx])


def check(P, psi, tol):
    nz, ny, nx = psi.shape
    s = P.Solver(nx, ny, nz, *H, 0.01, g=9.0, prec="f32")
    s.set_psi(psi)
    n1, n2 = exact(psi)
    for a in range(3 if nz > 1 else 2):
        assert np.all(abs(s.density1d(a) - n1[a]) <= tol * n1[a]), a
    for a in range(3 if nz > 1 else 1):
        assert np.all(abs(s.density2d(a) - n2[a]) <= tol * n2[a]), a
    s.close()


def field(shape, cplx):
    rng = np.random.default_rng(sum(shape))
    psi = rng.standard_normal(shape[::-1])
    if cplx:
        psi = psi + 1j * rng.standard_normal(psi.shape)
    return psi.astype(np.complex64 if cplx else np.float32).astype(complex if cplx else float)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("shape", [(37, 29, 21), (130, 33, 1)])
def test_columns_far_below_their_neighbours(P, shape, cplx):
    """Neighbouring columns, and rows, 2^40 and 2^120 apart (one column all but subnormal).
    Tolerance 2^-40: the values, not the last bits, are looked at here."""
    psi = field(shape, cplx)
    size = np.array([1.0, 2.0 ** -40, 2.0 ** -70, 2.0 ** -120, 2.0 ** 30, 2.0 ** -100])
    psi = psi * size[np.arange(shape[0]) % 6][None, None, :]
    psi = (psi.astype(np.complex64) if cplx else psi.astype(np.float32)).astype(psi.dtype)
    check(P, psi, 2.0 ** -40)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("amp", [1.0, 2.0 ** 100, 2.0 ** 126, 2.0 ** -120])
@pytest.mark.parametrize("shape", [(37, 29, 21), (200, 70, 33), (130, 33, 1), (5, 3, 400), (3, 501, 7)])
def test_fp64_precision(P, shape, amp, cplx):
    psi = field(shape, cplx)
    psi = (np.clip(abs(psi.real), 0.01, 1.99) + (1j * np.clip(abs(psi.imag), 0.01, 1.99) if cplx else 0)) * amp
    psi = (psi.astype(np.complex64) if cplx else psi.astype(np.float32)).astype(psi.dtype)
    check(P, psi, 8 * 2.0 ** -53)
