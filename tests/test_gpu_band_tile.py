"""Banded y / z sweeps over shared-memory tiles: runs, parts of a line, position chunks and
their remainders on both axes, half-widths 3, 5 and 8, planes, single steps (a graph)
and timed (separate) launches, against the oracle.  Tolerance: the FP32 short-run bound of
44 roundings of 2^-24 per step and point, a random walk over them."""
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


SHAPES = [(8, 8, 8), (9, 44, 45), (128, 43, 88), (130, 57, 56), (133, 89, 11), (256, 9, 113), (40, 150, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("a", [0.004, 0.025, 0.06])
@pytest.mark.parametrize("mode", ["imag", "real"])
def test_runs_parts_and_chunks(P, orc, shape, a, mode):
    h, steps = 0.2, 5
    p = orc.Problem(*shape, h, 0.97 * h, 1.03 * h, 4 * a * h * h, gamma=1.0, nu=1.4, lam=1.9, g=20.0)
    psi = orc.init_gaussian(p)
    if mode == "real":
        x = (np.arange(shape[0]) - 0.5 * (shape[0] - 1)) * h
        psi = psi * np.exp(0.3j * np.sin(x))[None, None, :]
    ref = (orc.step_real if mode == "real" else orc.step_imag)(p, psi, steps)
    s = P.Solver(*shape, h, 0.97 * h, 1.03 * h, 4 * a * h * h, 1.0, 1.4, 1.9, g=20.0, prec="f32")
    s.set_psi(psi)
    step = s.step_real if mode == "real" else s.step_imag
    step(2)
    step(1)
    P.gp_set_timing(s.handle, True)
    step(2)
    P.gp_set_timing(s.handle, False)
    got = s.get_psi(as_complex=mode == "real")
    # (a start rounded to FP32 costs one more rounding)
    assert np.max(np.abs(got - ref)) <= (steps * np.sqrt(44) + 1) * 2.0 ** -24 * np.max(np.abs(ref))
    s.close()
