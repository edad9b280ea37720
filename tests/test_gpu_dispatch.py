"""Which sweeps a solver runs (gp_get_info), at the edges of each rule: the FP64 increment form, the
FP32 sweeps over shared-memory tiles, the joined x and y sweep.  The tests of their results compare
with the oracle and would pass on any other kernel too."""
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


def facts(P, shape, prec, h, dt, mode):
    s = P.Solver(*shape, h, dt=dt, gamma=1.0, nu=1.41, lam=2.0, g=5.0, prec=prec)
    s.init_gaussian()
    if mode == "real":
        s.step_real(0)
    d = s.info()
    s.close()
    return d


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("shape,dt,mask", [
    ((64, 48, 32), 0.004, 7), ((45, 38, 34), 0.003, 7), ((16, 16, 16), 0.004, 7), ((2048, 16, 17), 0.004, 7),
    ((15, 40, 40), 0.004, 6), ((40, 15, 40), 0.004, 5), ((64, 48, 15), 0.004, 3), ((50, 40, 1), 0.004, 3),
    ((64, 48, 32), 0.16 * 0.03125, 7), ((64, 48, 32), 0.16 * 0.0313, 0)])
def test_increment_form(P, shape, dt, mask, mode):
    d = facts(P, shape, "f64", 0.2, dt, mode)
    assert d["line64_mask"] == 7 and d["inc64_mask"] == mask


@pytest.mark.parametrize("shape,dt,imag,real", [
    ((131, 97, 61), 0.004, 6, 6), ((300, 256, 1), 0.004, 2, 2), ((8, 8, 8), 0.004, 6, 6), ((133, 89, 11), 0.0096, 6, 6),
    ((240, 200, 160), 0.004, 6, 0), ((300, 240, 200), 0.004, 2, 0), ((64, 7, 32), 0.004, 4, 4)])
def test_tiles(P, shape, dt, imag, real):
    assert facts(P, shape, "f32", 0.2, dt, "imag")["tile_mask"] == imag
    assert facts(P, shape, "f32", 0.2, dt, "real")["tile_mask"] == real


@pytest.mark.parametrize("mode", ["imag", "real"])
@pytest.mark.parametrize("shape,dt,joined", [
    ((64, 48, 32), 0.004, 1), ((64, 48, 32), 0.0008, 1), ((8, 8, 8), 0.004, 1), ((256, 32, 64), 0.004, 1),
    ((257, 32, 32), 0.004, 0), ((256, 33, 64), 0.004, 0), ((24, 100, 80), 0.004, 0), ((64, 48, 32), 0.0096, 0),
    ((300, 256, 1), 0.004, 0)])
def test_joined_sweep(P, shape, dt, joined, mode, monkeypatch):
    if dt == 0.0096 and mode == "real":
        pytest.skip("half-width 5 there")
    assert facts(P, shape, "f32", 0.2, dt, mode)["xy"] == joined
    monkeypatch.setenv("GP_XY", "0")
    assert facts(P, shape, "f32", 0.2, dt, mode)["xy"] == 0
