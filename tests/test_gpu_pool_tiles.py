"""Batched y / z sweeps over shared-memory tiles (k_batch_tile) and the two modes side by side,
against the oracle: lines of 8 points (one run per block), of one point more and less than the
run limits (11 and 14 points per run; 1, 2 and 4 runs), rows narrower than a vector's multiple,
every runs setting, single steps and runs of steps.  Tolerance: the FP32 short-run bound of
test_gpu_pool.py, 3e-6 of the field's maximum.
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


LINES = [(9, 8, 8), (16, 11, 12), (21, 13, 14), (32, 22, 25), (10, 44, 45), (13, 23, 57), (48, 9, 16)]


@pytest.mark.parametrize("turns", [1, 2, 3])
@pytest.mark.parametrize("dt", [0.004, 0.0008])   # imaginary time: W = 5, W = 3
def test_pool_tiles_against_the_oracle(P, orc, turns, dt):
    h, steps = 0.2, (1, 2, 17)
    pool = P.Pool(64 << 20, max_slots=2 * len(LINES))
    pool.set_shape(3, turns)
    slots = [(pool.add(nx=x, ny=y, nz=z, dx=h, dt=dt, gamma=1.0, nu=1.41, lam=2.0, g=5.0), (x, y, z), real)
             for real in (False, True) for x, y, z in LINES]
    for s, _, real in slots:
        if real:
            pool.set_real_time(s)
    for n in steps:
        pool.step(n)
    for s, (x, y, z), real in slots:
        p = orc.Problem(x, y, z, h, h, h, dt, gamma=1.0, nu=1.41, lam=2.0, g=5.0)
        psi = orc.init_gaussian(p)
        ref = orc.step_real(p, psi.astype(complex), sum(steps)) if real else orc.step_imag(p, psi, sum(steps))
        got = pool.get_psi(s, as_complex=real)
        assert np.max(np.abs(got - ref)) <= 3e-6 * np.max(np.abs(ref)), (x, y, z, real)
    pool.close()
