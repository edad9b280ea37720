"""Pools of long, thin slots: every half-width and runs setting, where the z sweep's blocks (columns
and runs rounded up apart) are many for the slot's size, a tuned pool among them.  Tolerance: the
FP32 short-run bound of test_gpu_pool.py, 3e-6 of the field's maximum."""
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


@pytest.mark.parametrize("shape", [(9, 8, 680), (9, 43, 120), (9, 22, 232), (8, 8, 712), (17, 8, 2048)])
@pytest.mark.parametrize("dt", [0.0008, 0.004, 0.0096])   # W = 3, 5, 8
def test_thin_slots(P, orc, shape, dt):
    h, steps = 0.2, 3
    p = orc.Problem(*shape, h, h, h, dt, gamma=1.0, nu=1.41, lam=0.05, g=5.0)
    ref = orc.step_imag(p, orc.init_gaussian(p), steps)
    for turns in (None, 1, 2, 3, "tune"):
        pool = P.Pool(64 << 20, max_slots=4)
        if turns in (1, 2, 3):
            pool.set_shape(3, turns)
        slot = pool.add(nx=shape[0], ny=shape[1], nz=shape[2], dx=h, dt=dt, gamma=1.0, nu=1.41, lam=0.05, g=5.0)
        if turns == "tune":
            pool.tune(2)
        pool.step(steps)
        got = pool.get_psi(slot)
        pool.close()
        assert np.max(np.abs(got - ref)) <= 3e-6 * np.max(np.abs(ref)), turns
