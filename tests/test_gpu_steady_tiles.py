"""Steady solver at the edges of its tiles: the first-order residual (8 x 6 cells per CTA below 100k cells,
32 x 15 above) with the local steps it computes, and LU-SGS sweeps on whole, ragged and single-row tiles,
against the oracle with the tolerances of the parity tests of the steady solver (1e-12 and 1e-11 of the
largest value in double precision)."""
import numpy as np
import pytest

from test_gpu_steady import both, corner, rel, wavy

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


@pytest.mark.parametrize("n", [(8, 6), (9, 7), (17, 13), (16, 5), (400, 256)])
@pytest.mark.parametrize("turb", [0, 2])
def test_first_order_residual(n, turb):
    sp = wavy(n[0], n[1], seed=sum(n), turb=turb)
    s, c, W, f1, f2 = both(sp, levels=1)
    dt_g, R_g = s.residual(cfl_flux=0.5, first_order=True)
    dt_o, R_o = c.steady_residual(sp["nodes"], W, cfl_flux=0.5, first_order=True, f1=f1, f2=f2, nthreads=8)
    assert rel(dt_g, dt_o) < 1e-13
    nc = W.size // 4
    for v in range(4):
        a, b = R_g[v * nc:(v + 1) * nc], R_o[v * nc:(v + 1) * nc]
        assert np.abs(a - b).max() < 1e-12 * np.abs(b).max() + 1e-15
    s.close()


@pytest.mark.parametrize("n", [(16, 16), (17, 16), (16, 17), (15, 33), (40, 3)])
@pytest.mark.parametrize("tile", [16, 32])
def test_lusgs_sweeps(n, tile):
    sp = corner(n[0], n[1], turb=0)
    s, c, W, f1, f2 = both(sp, levels=1, tile=tile)
    s.cycles(2, cfl=3.0, cfl_flux=0.5)
    Wo = W
    for _ in range(2):
        Wo, _, st = c.steady_cycle(sp["nodes"], Wo, 3.0, cfl_flux=0.5, levels=1, tiles=(tile, tile), f1=f1, f2=f2,
                                   nthreads=8)
        assert st == 0
    Wg = s.get_state()
    nc = W.size // 4
    for v in range(4):
        a, b = Wg[v * nc:(v + 1) * nc], Wo[v * nc:(v + 1) * nc]
        assert np.abs(a - b).max() < 1e-11 * np.abs(b).max()
    s.close()
