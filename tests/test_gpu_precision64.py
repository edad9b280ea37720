"""FP64 steps against the same steps in extended precision (numpy's long double): fields on
which arithmetic in two FP32 parts has no bits to spare.

Tolerance: a step is four substeps, and whichever way a substep is evaluated its relative L2
error is to stay within 2^-53, that of the FP64 operations it replaces (an FP64 recurrence or
product of factors measures 0.9e-16..1.2e-16); the substeps' roundings are independent:
sqrt(4 steps) 2^-53.  (The renormalisation factor of imaginary time, which all points share, is an
FP64 sum over the field with a rounding error of its own: it is divided out.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
W = (1.0, 1.41, 2.0)


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1605_03958_gb300 as pkg
    return pkg


def solve(u, axis, a):
    """(I + aK)^-1 (I - aK) u along an axis, K the second difference with zero ghosts."""
    u = np.moveaxis(u, axis, 0)
    n = u.shape[0]
    r = (1 - 2 * a) * u
    r[1:] += a * u[:-1]
    r[:-1] += a * u[1:]
    c = np.empty(n, u.dtype)
    for j in range(n):
        den = 1 + 2 * a + (a * c[j - 1] if j else 0)
        c[j] = -a / den
        r[j] = (r[j] + (a * r[j - 1] if j else 0)) / den
    for j in range(n - 2, -1, -1):
        r[j] -= c[j] * r[j + 1]
    return np.moveaxis(r, 0, axis)


def exact(shape, h, dt, g, mode, psi, steps):
    Q = np.longdouble
    u = psi.astype(np.clongdouble if mode == "real" else Q)
    x, y, z = ((np.arange(n) - Q(0.5) * (n - 1)) * Q(h) for n in shape)
    V = sum(Q(w) ** 2 / 2 * q * q for w, q in zip(W, (x[None, None, :], y[None, :, None], z[:, None, None])))
    a = Q(dt) / (4 * Q(h) * Q(h)) * (1j if mode == "real" else 1)
    axes = (2, 1) if shape[2] == 1 else (2, 1, 0)
    for _ in range(steps):
        d = Q(dt) * (V + Q(g) * (u.real * u.real + (u.imag * u.imag if mode == "real" else 0)))
        u = u * (np.cos(d) - 1j * np.sin(d) if mode == "real" else np.exp(-d))
        for ax in axes:
            u = solve(u, ax, a)
        if mode == "imag":
            u = u / np.sqrt((u * u).sum() * Q(h) ** len(axes))
    return u


def check(P, shape, h, dt, g, mode, psi, steps):
    s = P.Solver(*shape, h, dt=dt, gamma=W[0], nu=W[1], lam=W[2], g=g, prec="f64")
    s.set_psi(psi)
    (s.step_real if mode == "real" else s.step_imag)(steps)
    got = s.get_psi(as_complex=mode == "real")
    s.close()
    ref = exact(shape, h, dt, g, mode, psi, steps)
    if mode == "imag":
        got = got.astype(np.longdouble)
        got = got * ((got * ref).sum() / (got * got).sum())
    err = float(np.sqrt((abs(got - ref) ** 2).sum() / (abs(ref) ** 2).sum()))
    assert err <= np.sqrt(4 * steps) * 2.0 ** -53, err


def noise(shape, mode, seed=3):
    rng = np.random.default_rng(seed)
    f = 0.3 * rng.standard_normal(shape[::-1])
    return f + 0.3j * rng.standard_normal(f.shape) if mode == "real" else f


@pytest.mark.parametrize("shape", [(512, 304, 1), (512, 64, 9)])
def test_noise_in_a_field_that_has_fallen(P, shape):
    """Grids without an increment sweep along z (planes, nz < 16), noise 2^20 above its
    normalised size at the start: what counts as noise follows the field down."""
    h = 0.05   # (a trap whose factor stays near 1 over the whole grid)
    check(P, shape, h, 0.1 * h * h, 0.0, "imag", noise(shape, "imag") * 2.0 ** 20, 3)


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("amp", [2.0 ** -85, 2.0 ** -95, 1e-45, 1e-60, 1e-150])
@pytest.mark.parametrize("shape", [(45, 38, 34), (64, 50, 1)])
def test_fields_of_very_small_amplitude(P, mode, amp, shape):
    """At the edge of FP32's exponent range and far below it; in imaginary time the step after
    the first is of normal size again."""
    h, steps = 0.2, 2
    x, y, z = ((np.arange(n) - 0.5 * (n - 1)) * h for n in shape)
    f = amp * np.exp(-0.3 * (z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2))
    f = f * (1 + 0.2 * np.cos(1.3 * x + 0.4)[None, None, :] * np.cos(0.7 * y)[None, :, None])
    if mode == "real":
        f = f * np.exp(0.4j * np.sin(x + 0.2))[None, None, :]
    check(P, shape, h, 0.004, 0.0, mode, f, steps)


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("y,h", [(0.006, 0.05), (0.02, 0.05), (0.05, 0.05), (0.1, 0.05), (0.4, 0.05),
                                 (0.001, 0.2), (0.001, 0.3), (0.001, 0.45), (0.02, 0.3)])
@pytest.mark.parametrize("shape", [(45, 38, 34), (64, 50, 1)])
def test_substep_of_large_density_or_trap(P, shape, y, h, mode):
    """Fields spread over the whole box (half waves that vanish at its walls): dt g |psi|^2 up to
    y, trap factors from near 1 (h = 0.05) to exp(-2) and beyond at the walls (h = 0.45)."""
    s = [np.sin(np.pi * (np.arange(n) + 1) / (n + 1)) if n > 1 else np.ones(1) for n in shape]
    f = 0.3 * s[2][:, None, None] * s[1][None, :, None] * s[0][None, None, :]
    if mode == "real":
        f = f * np.exp(0.4j * np.sin(np.arange(shape[0]) * 0.1))[None, None, :]
    dt = 0.1 * h * h
    check(P, shape, h, dt, y / (0.09 * dt), mode, f, 1)


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("dtf", [0.05, 0.1, 0.125])
@pytest.mark.parametrize("shape", [(61, 50, 41), (32, 24, 24), (18, 17, 300), (90, 75, 1), (30, 16, 17)])
def test_noise_and_short_waves(P, shape, dtf, mode, request):
    """Grid-scale noise, and waves of seven points on a condensate: blocks of every size, from
    less than a warp's segments up."""
    if shape[2] == 300 and mode == "real":
        request.applymarker(pytest.mark.xfail(reason="trap phases of up to 9 rad at z = 30: rounding "
                                                     "the phase itself to FP64 is an error of 4e-16"))
    h = 0.2
    check(P, shape, h, dtf * h * h, 1.0, mode, noise(shape, mode), 1)
    x, y, z = ((np.arange(n) - 0.5 * (n - 1)) * h for n in shape)
    f = 0.3 * np.exp(-0.3 * (z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2))
    f = f * np.cos(0.9 * (z[:, None, None] + y[None, :, None] + x[None, None, :]) / h + 0.3)
    check(P, shape, h, dtf * h * h, 1.0, mode, f.astype(complex) if mode == "real" else f, 1)
