"""The first-order residual above 100k cells (16 x 11 cells per CTA) on whole and ragged tiles, against the oracle with
the tolerances of the parity tests of the steady solver."""
import numpy as np
import pytest

from test_gpu_steady import both, rel, wavy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(400, 253), (401, 254), (415, 242)])
def test_first_order_residual(n):
    sp = wavy(n[0], n[1], seed=sum(n), turb=2)
    s, c, W, f1, f2 = both(sp, levels=1)
    dt_g, R_g = s.residual(cfl_flux=0.5, first_order=True)
    dt_o, R_o = c.steady_residual(sp["nodes"], W, cfl_flux=0.5, first_order=True, f1=f1, f2=f2, nthreads=8)
    assert rel(dt_g, dt_o) < 1e-13
    nc = W.size // 4
    for v in range(4):
        a, b = R_g[v * nc:(v + 1) * nc], R_o[v * nc:(v + 1) * nc]
        assert np.abs(a - b).max() < 1e-12 * np.abs(b).max() + 1e-15
    s.close()
