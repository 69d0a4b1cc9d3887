"""gks_face_flux at the ends of its arguments' ranges: an infinite centre-to-face distance (a side without a gradient
towards the face), and a time step that is subnormal in single precision."""
import numpy as np
import pytest

import oracle
from test_gpu_face_records import records

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1302_2132_gb300 import gks  # noqa: E402


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32", 1e-5)])  # the bars of the parity tests
@pytest.mark.parametrize("sides", [(0,), (1,), (0, 1)])
def test_infinite_distance(sides, precision, tol):
    rec = records(2, 20, 9)
    rec[:, [32 + s for s in sides]] = np.inf
    F, _ = gks.face_flux(2, torch.tensor(rec, device="cuda"), 1e-3, mu=1e-4, C_a=0.3, precision=precision)
    F = F.cpu().numpy()
    for i, r in enumerate(rec):
        f = oracle.make_face(2, r[:4], r[4:8], r[8:12], r[12:16], r[16:20], r[20:24], r[24:28][None], r[28:32][None],
                             r[32], r[33], r[34])
        Fo = oracle.face_flux(2, 1.4, 1e-4, 0.3, 1e-3, f, multid=1)
        assert np.linalg.norm(F[i] - Fo) <= tol * np.linalg.norm(Fo)


@pytest.mark.parametrize("D", [1, 2, 3])
def test_subnormal_time_step(D):
    """Without viscosity the flux is dt times the Euler flux of the face: 60 operations, each within half the subnormal
    spacing (7e-46) or 2^-23 of the largest value."""
    rec = torch.tensor(records(D, 40, 3), device="cuda")
    rec[:, -1] = 0.0
    out = [gks.face_flux(D, rec, 5e-39, mu=0.0, C_a=0.0, precision=p)[0].cpu().numpy() for p in ("fp64", "fp32")]
    assert np.isfinite(out[1]).all()
    assert np.abs(out[1] - out[0]).max() <= 60 * (7.1e-46 + 2.0 ** -23 * np.abs(out[0]).max())
