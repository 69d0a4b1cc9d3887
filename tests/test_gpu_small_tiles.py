"""The tiles of small grids (8 x 8 cells in 2D, 30 in 1D) at their edges: grids of less than a tile, of whole tiles
and one cell more, in every boundary kind of the parity cases, against the oracle (FP64, the 1e-12 per step of
the parity tests), and in single precision against the 32 x 15 tile to its rounding.  Consecutive steps
are launched as programmatic dependents here, so a run of many steps is compared as well."""
import numpy as np
import pytest

import oracle
from cases import gpu_solver, max_rel_elementwise, oracle_case, rel_err_per_var
from paper_1302_2132_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def flow(n, kind):
    rng = np.random.default_rng(sum(n))
    D = len(n)
    prim = 1.0 + 0.1 * rng.random((D + 2,) + n[::-1])
    bc = {"periodic": [[0, 0]] * D, "mixed": [[2, 1], [4, 2]][:D]}[kind]
    s = dict(dim=D, n=n, dx=[rng.uniform(0.8, 1.2, k) for k in n], bc=bc, prim=prim, T_wall=1.0)
    s["f1"], s["f2"] = (rng.uniform(0.01, 0.02, n[::-1]) for _ in range(2))
    return s


@pytest.mark.parametrize("n,variant", [((3, 5), "9"), ((8, 8), "9"), ((9, 16), "9"), ((17, 7), "9"), ((5,), "3"),
                                       ((30,), "3"), ((31,), "3"), ((61,), "3")])
@pytest.mark.parametrize("kind", ["periodic", "mixed"])
def test_fp64_steps(monkeypatch, n, variant, kind):
    monkeypatch.setenv("GKS_TILE_VARIANT", variant)
    spec = flow(n, kind)
    kw = dict(turb_model=2, multid=int(len(n) > 1), mu=1e-3, C_a=0.4)
    s, c = gpu_solver(spec, **kw), oracle_case(spec, **kw)
    s.set_state(spec["prim"].ravel(), layout="soa_prim")
    s.set_turbulence(spec["f1"].ravel(), spec["f2"].ravel())
    s.step(nsteps=3, cfl=0.4)
    assert s.tile_shape()[0] == int(variant)
    W, _, _, st = c.run(c.prim_to_cons(spec["prim"].ravel()), 3, cfl=0.4, f1=spec["f1"].ravel(), f2=spec["f2"].ravel(),
                        nthreads=4)
    assert st == 0
    assert np.all(max_rel_elementwise(s.get_state(), W, len(n) + 2, 1e-2) < 3e-12)
    s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
@pytest.mark.parametrize("n", [(9, 16), (64, 40)])
def test_single_precision_matches_the_first_tile(monkeypatch, n, precision):
    out = []
    for v in ("0", "9"):
        monkeypatch.setenv("GKS_TILE_VARIANT", v)
        spec = flow(n, "mixed")
        s = gpu_solver(spec, turb_model=2, mu=1e-3, precision=precision)
        s.set_state(spec["prim"].ravel(), layout="soa_prim")
        s.set_turbulence(spec["f1"].ravel(), spec["f2"].ravel())
        s.step(nsteps=60, cfl=0.4)
        assert s.tile_shape()[0] == int(v)
        out.append(s.get_state())
        s.close()
    assert np.all(rel_err_per_var(out[1], out[0], 4) < 1e-6)
