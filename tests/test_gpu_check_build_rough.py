"""The bounds-checked build (-DGP_CHECK) on fields that FP64 increment sweeps compute in FP64:
noise (every block rough) and very small amplitudes.  No check fires and the results are the
normal build's bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_1605_03958_gb300 as P
out = []
for shape in [(16, 17, 16), (37, 29, 33), (301, 16, 20), (33, 65, 5), (40, 37, 1)]:
    for amp in (0.3, 1e-60):
        rng = np.random.default_rng(5)
        f = amp * rng.standard_normal(shape[::-1])
        s = P.Solver(*shape, 0.3, 0.25, 0.4, 0.005, 1.1, 1.7, 0.6, g=1.0, prec="f64")
        s.set_psi(f)
        s.step_imag(2)
        out.append(s.get_psi())
        s.set_psi(f * np.exp(1j))
        s.step_real(2)
        out.append(s.get_psi(as_complex=True))
        s.sync()
        s.close()
np.savez(sys.argv[2], *out)
"""


def test_rough_and_tiny_fields(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_1605_03958_gb300 import build
    got = []
    for name, lib in (("checked", build.build(check=True)), ("normal", build.LIB)):
        path = str(tmp_path / (name + ".npz"))
        r = subprocess.run([sys.executable, "-c", CHILD, ROOT, path], env=dict(os.environ, GP_SSCN_LIB=lib),
                           capture_output=True, text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]   # (a GP_ERR_BOUNDS fails the child)
        with np.load(path) as z:
            got.append([z[k] for k in z.files])
    assert len(got[0]) == 20
    for a, b in zip(*got):
        assert np.array_equal(a, b)
