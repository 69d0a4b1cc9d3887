"""Residual norms of the last step (gks_residual) against the same norms of the copied-out states, in
every precision, from grids smaller than one thread block to larger than one sweep of the
reduction's grid, on rectilinear and body-fitted grids."""
import numpy as np
import pytest

from cases import gpu_solver
from paper_1302_2132_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32_acc64"])
@pytest.mark.parametrize("n,curved", [((5,), False), ((257,), False), ((33, 17), False), ((480, 400), False),
                                      ((7, 5, 9), False), ((40, 23), True)])
def test_residual_norms_of_the_states(n, curved, precision):
    rng = np.random.default_rng(sum(n))
    D = len(n)
    prim = 1.0 + 0.1 * rng.random((D + 2,) + n[::-1])
    dx = [rng.uniform(0.5, 1.5, k) for k in n]
    s = gpu_solver(dict(dim=D, n=n, dx=dx, bc=[[0, 0]] * D, prim=prim), precision=precision, mu=1e-3,
                   multid=0 if curved else 1)
    vol = np.ones(n[::-1])
    for d in range(D):
        vol = vol * dx[d].reshape([-1 if a == D - 1 - d else 1 for a in range(D)])
    if curved:
        nodes = inputs.wavy_nodes(*n)
        s.set_nodes(nodes)
        d1, d2 = nodes[1:, 1:] - nodes[:-1, :-1], nodes[1:, :-1] - nodes[:-1, 1:]
        vol = 0.5 * (d1[..., 0] * d2[..., 1] - d2[..., 0] * d1[..., 1])
    s.set_state(prim.ravel(), layout="soa_prim")
    dt = s.compute_dt(0.3)
    s.step(nsteps=3, dt=dt)
    W0 = s.get_state().reshape(D + 2, -1)
    s.step(nsteps=1, dt=dt)
    W1 = s.get_state().reshape(D + 2, -1)
    l2, linf, total = s.residual()
    r = (W1 - W0) / dt
    # double states: the same differences, so only the order of the sums differs (n eps); float pairs: the
    # difference of two pairs is formed in single precision (three roundings of 2^-24)
    tol = 4 * 2.0 ** -24 if precision == "fp32" else 1e-12
    assert np.allclose(l2, np.sqrt((r * r).mean(1)), rtol=tol, atol=0)
    assert np.allclose(linf, np.abs(r).max(1), rtol=tol, atol=0)
    assert np.allclose(total, (W1 * vol.ravel()).sum(1), rtol=1e-12, atol=0)
    s.close()
