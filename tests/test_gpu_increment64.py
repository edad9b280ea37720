"""FP64 sweeps in increment form (lines of at least 16 points, a = dt / (4 h^2) <= 1/32)
against the oracle: segment edges on every axis, odd row lengths and row counts, a just
inside and outside the rule, grid-scale noise (evaluated in FP64), amplitudes far outside
FP32's range, long and short nonlinear sums and trap factors far from 1.

Tolerance: per step and side at most 8 roundings of 2^-53 max|psi| in each of the three
sweeps and 8 in the pointwise substep, added linearly over the steps and over the two
sides: 64 steps 2^-53 max|psi|."""
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


def compare(P, orc, shape, h, dt, g, mode, psi0, steps=4, w=(1.0, 1.41, 2.0)):
    p = orc.Problem(*shape, h, h, h, dt, gamma=w[0], nu=w[1], lam=w[2], g=g)
    ref = (orc.step_real if mode == "real" else orc.step_imag)(p, psi0, steps)
    s = P.Solver(*shape, h, dt=dt, gamma=w[0], nu=w[1], lam=w[2], g=g, prec="f64")
    s.set_psi(psi0)
    (s.step_real if mode == "real" else s.step_imag)(steps)
    got = s.get_psi(as_complex=mode == "real")
    s.sync()
    s.close()
    scale = max(np.max(np.abs(ref)), np.max(np.abs(psi0)) if mode == "real" else 0.0)
    assert np.max(np.abs(got - ref)) <= 64 * steps * 2.0 ** -53 * scale


def smooth(shape, h, mode, amp=0.3):
    nx, ny, nz = shape
    x, y, z = ((np.arange(n) - 0.5 * (n - 1)) * h for n in shape)
    f = amp * np.exp(-0.3 * (z[:, None, None] ** 2 + y[None, :, None] ** 2 + x[None, None, :] ** 2))
    f = f * (1 + 0.2 * np.cos(1.3 * x + 0.4)[None, None, :] * np.cos(0.7 * y)[None, :, None])
    return f * np.exp(0.4j * np.sin(x + 0.2))[None, None, :] if mode == "real" else f


SHAPES = [(16, 17, 16), (17, 16, 33), (31, 32, 15), (33, 49, 24), (64, 15, 47), (240, 20, 18), (523, 16, 16),
          (18, 600, 16), (16, 17, 1100), (2048, 16, 17), (50, 40, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mode", ["imag", "real"])
def test_segment_edges(P, orc, shape, mode):
    compare(P, orc, shape, 0.2, 0.004, 40.0, mode, smooth(shape, 0.2, mode))


@pytest.mark.parametrize("a", [1.0 / 32, 1.0 / 32 * (1 + 1e-12), 1e-9])
@pytest.mark.parametrize("mode", ["imag", "real"])
def test_edges_of_the_rule(P, orc, a, mode):
    h = 0.2
    compare(P, orc, (37, 33, 29), h, 4 * a * h * h, 10.0, mode, smooth((37, 33, 29), h, mode))


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("kind", ["noise", "large", "tiny"])
def test_noise_and_range(P, orc, mode, kind):
    shape = (45, 38, 34)
    rng = np.random.default_rng(3)
    f = 0.3 * rng.standard_normal((shape[2], shape[1], shape[0]))
    if mode == "real":
        f = f + 0.3j * rng.standard_normal(f.shape)
    if kind != "noise":
        f = smooth(shape, 0.2, mode) * (1e25 if kind == "large" else 1e-30)
    compare(P, orc, shape, 0.2, 0.003, 20.0 if kind == "noise" else 0.0, mode, f)


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("g,h", [(0.5, 0.2), (30.0, 0.2), (90.0, 0.2), (170.0, 0.2), (400.0, 0.2), (5.0, 0.9)])
def test_pointwise_branches(P, orc, mode, g, h):
    """dt g max|psi|^2 from 2e-4 to 0.14 at h = 0.2 (short and long sums, their doublings,
    FP64); at h = 0.9 trap factors down to exp(-9) in a box of 40 oscillator lengths."""
    shape = (44, 40, 36)
    compare(P, orc, shape, h, 0.1 * h * h if h < 0.5 else 0.02, g, mode, smooth(shape, h, mode), steps=2)


def test_zero_field_is_reported(P):
    s = P.Solver(32, 24, 20, 0.2, dt=0.004, g=5.0, prec="f64")
    s.set_psi(np.zeros((20, 24, 32)))
    s.step_imag(1)
    with pytest.raises(P.GPError) as e:
        s.sync()
    assert e.value.code == P.gp.GP_ERR_NONFINITE
    s.close()
