"""gks_face_flux reads its records through shared memory in CTAs of 64 faces: counts round the CTA size and
records that start on an 8-byte (not 16-byte) boundary give the fluxes of the same faces one by one, and a record
in single precision is the rounded record."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1302_2132_gb300 import gks  # noqa: E402


def records(D, n, seed):
    rng = np.random.default_rng(seed)
    nv = D + 2
    rec = rng.normal(size=(n, gks.face_record_len(D)))
    for o in range(4):  # wl, wr, cl, cr
        rho, U, p = rng.uniform(0.5, 2, n), rng.uniform(-1, 1, (n, D)), rng.uniform(0.5, 2, n)
        rec[:, o * nv:(o + 1) * nv] = np.concatenate(
            [rho[:, None], rho[:, None] * U, (p / 0.4 + 0.5 * rho * (U * U).sum(1))[:, None]], 1)
    rec[:, -3:-1] = rng.uniform(0.01, 0.02, (n, 2))
    rec[:, -1] = rng.uniform(0, 1e-3, n)
    rec[::7, 4 * nv] = 0.0  # zeros and values that are subnormal in single precision
    rec[::5, 4 * nv + 1] = 1e-41
    return rec


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 129])
@pytest.mark.parametrize("offset", [0, 1])
def test_counts_and_alignment(D, n, offset, precision):
    rec = records(D, n, 100 * D + n)
    flat = torch.zeros(rec.size + 2, dtype=torch.float64, device="cuda")
    part = flat[offset:offset + rec.size].view(n, -1)
    part.copy_(torch.tensor(rec))
    assert part.data_ptr() % 16 == 8 * offset
    F, tau = gks.face_flux(D, part, 1e-3, mu=1e-4, C_a=0.3, precision=precision)
    for i in range(n):
        Fi, ti = gks.face_flux(D, part[i:i + 1].clone(), 1e-3, mu=1e-4, C_a=0.3, precision=precision)
        assert torch.equal(F[i], Fi[0]) and tau[i] == ti[0]
    if precision == "fp32":
        Fr, _ = gks.face_flux(D, part.float().double(), 1e-3, mu=1e-4, C_a=0.3, precision=precision)
        assert torch.equal(F, Fr)


@pytest.mark.parametrize("mach", [0.0, 1e-9, 0.3, 1.0, 3.0, 8.0])
@pytest.mark.parametrize("sign", [-1.0, 1.0])
def test_fp64_flux_over_the_range_of_the_half_line_moments(mach, sign):
    """Both sides at the same normal Mach number, from rest (erfc near 1) to far supersonic (one half line empty):
    the double flux matches the oracle to the 1e-12 of the parity tests."""
    import oracle
    D, nv, n, dt = 2, 4, 20, 1e-3
    rng = np.random.default_rng(int(10 * mach) + 7)
    rec = records(D, n, 5)
    for o in range(4):
        rho, p = rng.uniform(0.5, 2, n), rng.uniform(0.5, 2, n)
        u = np.stack([sign * mach * np.sqrt(1.4 * p / rho), rng.uniform(-1, 1, n)], 1)
        rec[:, o * nv:(o + 1) * nv] = np.concatenate(
            [rho[:, None], rho[:, None] * u, (p / 0.4 + 0.5 * rho * (u * u).sum(1))[:, None]], 1)
    F, _ = gks.face_flux(D, torch.tensor(rec, device="cuda"), dt, mu=1e-4, C_a=0.3, precision="fp64")
    F = F.cpu().numpy()
    for i in range(n):
        r = rec[i]
        f = oracle.make_face(D, r[:4], r[4:8], r[8:12], r[12:16], r[16:20], r[20:24], r[24:28][None], r[28:32][None],
                             r[32], r[33], r[34])
        Fo = oracle.face_flux(D, 1.4, 1e-4, 0.3, dt, f, multid=1)
        assert np.linalg.norm(F[i] - Fo) <= 1e-12 * np.linalg.norm(Fo)
