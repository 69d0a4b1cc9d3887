"""Residual norms of the float-pair form are those of the stored states in double, also where a step changes a state by
less than single precision resolves.  Differences and sums in double: only the order of the sums differs (n eps)."""
import numpy as np
import pytest

from cases import gpu_solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(100,), (40, 30), (12, 9, 8)])
@pytest.mark.parametrize("amplitude", [0.1, 1e-6])
def test_float_pair_norms(n, amplitude):
    rng = np.random.default_rng(sum(n))
    D = len(n)
    prim = 1.0 + amplitude * rng.random((D + 2,) + n[::-1])
    s = gpu_solver(dict(dim=D, n=n, dx=[np.ones(k) for k in n], bc=[[0, 0]] * D, prim=prim), precision="fp32", mu=1e-3,
                   multid=int(D > 1))
    s.set_state(prim.ravel(), layout="soa_prim")
    dt = s.compute_dt(0.3)
    s.step(nsteps=1, dt=dt)
    W0 = s.get_state().reshape(D + 2, -1)
    s.step(nsteps=1, dt=dt)
    W1 = s.get_state().reshape(D + 2, -1)
    l2, linf, _ = s.residual()
    r = (W1 - W0) / dt
    assert np.allclose(l2, np.sqrt((r * r).mean(1)), rtol=1e-12, atol=0)
    assert np.allclose(linf, np.abs(r).max(1), rtol=1e-12, atol=0)
    s.close()
