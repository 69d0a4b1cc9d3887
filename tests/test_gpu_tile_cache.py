"""The tile shape found for one reconstruction is not handed to a solver with another on the same grid: a
single-precision MUSCL-2 solver, whose shapes are ten, steps first, then MUSCL-3 and WENO-5 solvers, whose kernels are
built for two.  Each takes a shape it has, and its steps are, to the last bit, those of a solver forced to
that shape."""
import numpy as np
import pytest

from paper_1302_2132_gb300 import inputs
from tests.cases import gpu_solver

pytestmark = pytest.mark.gpu


def two_steps(spec, recon, dt):
    s = gpu_solver(spec, turb_model=1, mu=1e-4, precision="fp32", recon=recon)
    s.set_state(np.asarray(spec["prim"], dtype=np.float64).ravel(), layout="soa_prim")
    s.set_turbulence(np.asarray(spec["f1"], dtype=np.float64).ravel(), np.asarray(spec["f2"], dtype=np.float64).ravel())
    s.step(nsteps=2, dt=dt)
    W, shape = s.get_state(), s.tile_shape()[0]
    s.close()
    return W, shape


@pytest.mark.parametrize("n", [40, 96, 150, 260, 420])
def test_reconstructions_one_after_another(monkeypatch, n):
    spec = inputs.turbulence(n, 2, seed=5)
    dt = 0.2 * float(np.min(spec["dx"][0]))
    two_steps(spec, 0, dt)
    for recon in (1, 2):
        W, shape = two_steps(spec, recon, dt)
        assert shape in (0, 3)
        with monkeypatch.context() as m:
            m.setenv("GKS_TILE_VARIANT", str(shape))
            V, forced = two_steps(spec, recon, dt)
        assert forced == shape and np.array_equal(W, V)
