"""Banded x and y sweeps in one launch (k_band_xy, small 3D FP32 grids) against the two
separate sweeps: the same operations in the same order, so the same bits, as long as a row
takes the short polynomial in both.  Rows of one lane and of all 32, ragged ends of every
length, blocks of one row and of twelve, planes with a single block (both images in reach),
half-widths 3 and 5, a row too wide for it, both modes and splittings, steps by the graph and by direct launches.
"""
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


SHAPES = [(8, 8, 8), (9, 13, 8), (15, 12, 9), (33, 25, 10), (37, 11, 8), (64, 48, 32), (100, 8, 20),
          (197, 37, 8), (199, 24, 9), (200, 32, 32), (255, 24, 9), (256, 32, 32),
          (257, 24, 8), (8, 8, 200)]


@pytest.mark.parametrize("shape", SHAPES + [(16 + r, 14, 8) for r in range(8)])
@pytest.mark.parametrize("hs", [(0.2, 0.21, 0.22), (0.5, 0.5, 0.5)])   # dt = 0.004: W = 5, W = 3
@pytest.mark.parametrize("real", [False, True])
def test_joined_sweeps_give_the_bits_of_separate_ones(P, shape, hs, real, monkeypatch):
    outs = []
    for flag in ("1", "0"):
        monkeypatch.setenv("GP_XY", flag)
        s = P.Solver(*shape, *hs, 0.004, 1.0, 1.41, 2.0, g=1.0, prec="f32")
        s.init_gaussian()
        s.step_imag(3)
        for scheme in ("lie", "strang"):
            s.set_splitting(scheme)
            for n in (1, 4):
                (s.step_real if real else s.step_imag)(n)
        outs.append(s.get_psi(as_complex=real))
        assert abs(s.observables()["norm"] - 1.0) <= 1e-5
        s.close()
    assert np.array_equal(outs[0], outs[1])
