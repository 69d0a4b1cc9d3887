"""k-omega transport in three dimensions with omega near its default floor (1e-12), where (beta* omega)^3 is below single
precision's normal range: the single-precision forms keep omega, as the FP64 form does.

Tolerance: per step a cell's omega takes fewer than 40 single-precision operations of order omega (six
face fluxes of four, the sources and the two quotients), each within 2^-23: 2 steps x 40 x 1.2e-7 < 1e-5."""
import numpy as np
import pytest

from paper_1302_2132_gb300 import inputs
from tests.cases import gpu_solver

pytestmark = pytest.mark.gpu


def transported(spec, omega, precision, dt):
    n = spec["prim"][0].size
    s = gpu_solver(spec, turb_model=4, mu=1e-5, precision=precision)
    s.set_state(np.asarray(spec["prim"], dtype=np.float64).ravel(), layout="soa_prim")
    s.set_turbulence(np.full(n, 1e-14), omega)
    s.step(nsteps=2, dt=dt)
    k, om = s.get_turbulence()
    s.close()
    return np.asarray(om, dtype=np.float64)


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
def test_omega_near_its_floor(uniform, precision):
    spec = inputs.turbulence(12, 3, seed=13)
    spec["prim"] = np.array(spec["prim"], dtype=np.float64)
    if uniform:  # no strain, no vorticity: omega decays by a part in 1e15
        spec["prim"][0], spec["prim"][1:4], spec["prim"][4] = 1.0, 0.1, 1.0 / 1.4
    # on both sides of 2.5e-12, below which the cube is subnormal, all above the floor
    omega = 1.5e-12 * 16.0 ** np.random.default_rng(3).random(spec["prim"][0].size)
    if uniform:
        omega[:] = 2e-12
    want = transported(spec, omega, "fp64", 2e-3)
    got = transported(spec, omega, precision, 2e-3)
    if uniform:
        assert np.abs(want / 2e-12 - 1).max() < 1e-12
    assert np.abs(got / want - 1).max() < 1e-5
