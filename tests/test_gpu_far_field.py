"""FP64 fields on grids much wider than the condensate: the x sweep's substep where the trap
factor is far from 1 and the nonlinear argument below 2^-56."""
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


@pytest.mark.parametrize("shape", [(37, 32, 29), (48, 40, 16)])
@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("h", [0.5, 0.6])
def test_far_field_takes_the_trap_factor_alone(P, orc, shape, mode, h):
    """Wide grids, dt V up to 5: the x sweep leaves the two-part substep where the factor is
    far from 1 and, with |psi|^2 negligible there, multiplies by it alone; g = 0 (everywhere
    negligible) and g = 40.  Tolerance: FP64 steps against the oracle, 1e-12 of the maximum
    (15 steps of about 30 rounded operations each, 2^-53 a piece: 5e-14)."""
    dt = 0.1 * h * h
    for g in (0.0, 40.0):
        p = orc.Problem(*shape, h, h, h, dt, gamma=1.0, nu=1.41, lam=2.0, g=g)
        s = P.Solver(*shape, h, dt=dt, gamma=1.0, nu=1.41, lam=2.0, g=g, prec="f64")
        s.init_gaussian()
        psi = orc.init_gaussian(p)
        if mode == "imag":
            s.step_imag(15)
            got, ref = s.get_psi(), orc.step_imag(p, psi, 15)
        else:
            s.step_real(15)
            got, ref = s.get_psi(as_complex=True), orc.step_real(p, psi.astype(complex), 15)
        s.close()
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), (shape, mode, h, g)
