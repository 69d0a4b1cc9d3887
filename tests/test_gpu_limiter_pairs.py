"""Single-precision steps whose slopes, states and fluxes lie together in shared memory (2D) and whose limiters run
two variables at a time (body-fitted grids), at the edges of their tiles, for both limiters and expansions,
against the FP64 form.

Tolerance, of the largest conserved value after two steps: a single-precision face flux is within 3e-6 of its scale on
such states (its bar in the face tests is 1e-5), a step at CFL 0.4 adds four of them at dt (|U| + c) / dx <= 0.4, so
2 x 4 x 0.4 x 3e-6 = 1e-5."""
import numpy as np
import pytest

from cases import gpu_solver
from paper_1302_2132_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def spec_of(n, bc, nodes=None):
    rng = np.random.default_rng(n[0] * 100 + n[1])
    dx = [rng.uniform(0.8, 1.2, k) for k in n]
    s = dict(dim=2, n=n, dx=dx, bc=bc, T_wall=1.0, nodes=nodes)
    if nodes is None:
        x, y = (2 * np.pi * (np.cumsum(d) - 0.5 * d) / d.sum() for d in dx)
        X, Y = np.meshgrid(x, y)
        s["prim"] = np.stack([1 + 0.15 * np.sin(X + 2 * Y), 0.3 * np.cos(2 * X - Y), 0.2 * np.sin(X) * np.cos(Y),
                              1 + 0.1 * np.cos(X - Y)])
        s["f1"], s["f2"] = 0.01 + 0.002 * np.sin(X), 0.02 + 0.004 * np.cos(Y)
    else:
        pts = inputs.cell_points(nodes)
        s["prim"] = inputs.smooth_state_at(pts, seed=7, amp=0.15)
        s["f1"], s["f2"] = inputs.positive_fields_at(pts, seed=8)
    return s


def two_steps(spec, dt, **kw):
    s = gpu_solver(spec, turb_model=2, mu=1e-3, C_a=0.3, **kw)
    if spec["nodes"] is not None:
        s.set_nodes(spec["nodes"])
    s.set_state(np.asarray(spec["prim"], dtype=np.float64).ravel(), layout="soa_prim")
    s.set_turbulence(np.asarray(spec["f1"], dtype=np.float64).ravel(), np.asarray(spec["f2"], dtype=np.float64).ravel())
    dt = s.compute_dt(0.4) if dt is None else dt
    s.step(nsteps=2, dt=dt)
    W = s.get_state()
    s.close()
    return W, dt


def compare(spec, precision, **kw):
    W, dt = two_steps(spec, None, precision="fp64", **kw)
    V, _ = two_steps(spec, dt, precision=precision, **kw)
    assert np.abs(V - W).max() < 1e-5 * np.abs(W).max()


@pytest.mark.parametrize("n", [(5, 4), (32, 27), (33, 28)])
@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("multid", [0, 1])
@pytest.mark.parametrize("precision,recon", [("fp32", 0), ("fp32_acc64", 0), ("fp32", 1), ("fp32", 2)])
def test_rectilinear(n, limiter, multid, precision, recon):
    compare(spec_of(n, [[2, 1], [0, 0]]), precision, limiter=limiter, multid=multid, recon=recon)


@pytest.mark.parametrize("n", [(6, 5), (16, 11), (17, 12)])
@pytest.mark.parametrize("limiter", [0, 1])
@pytest.mark.parametrize("multid", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
def test_body_fitted(n, limiter, multid, precision):
    nodes = inputs.wavy_nodes(n[0], n[1], amp=0.04, shear=0.05)
    compare(spec_of(n, [[0, 0], [1, 1]], nodes), precision, limiter=limiter, multid=multid)
