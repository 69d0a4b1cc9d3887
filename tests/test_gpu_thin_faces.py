"""Faces whose two sides separate so fast that the density between them is subnormal: the flux stays finite, and the
tiles that evaluate two faces per thread give what the tiles with one do.

The sides have density rho and move apart at z sqrt(2 theta): the density between them is rho erfc(z).  In single
precision (rho = 1e-17) it is between 3e-39 and 1.1e-38 for the z below, in double (rho = 1e-200) between 6e-309 and
2.1e-308; its reciprocal is a number there."""
import numpy as np
import pytest

from paper_1302_2132_gb300 import gks
from tests.cases import gpu_solver

pytestmark = pytest.mark.gpu


def one_step(monkeypatch, D, variant, precision):
    monkeypatch.setenv("GKS_TILE_VARIANT", variant)
    n = (64, 24) if D == 2 else (32, 8, 8)
    rng = np.random.default_rng(D)
    z = rng.uniform(6.765, 6.856, n[::-1][:-1])[..., None]
    left = np.arange(n[0]) < n[0] // 2
    u = z * np.sqrt(2.0 / 1.4) * np.where(left, -1.0, 1.0)
    one = np.ones(n[::-1])
    prim = 1e-17 * np.stack([one, u * 1e17] + [0 * one] * (D - 1) + [one / 1.4])
    spec = dict(dim=D, n=n, dx=[np.ones(k) for k in n], bc=[[1, 1]] * D)
    s = gpu_solver(spec, mu=0.0, precision=precision)
    s.set_state(prim.ravel(), layout="soa_prim")
    s.step(nsteps=1, cfl=0.4)
    assert s.tile_shape()[0] == int(variant)
    W = s.get_state().reshape(D + 2, -1)
    s.close()
    return W


@pytest.mark.parametrize("precision", ["fp32", "fp32_acc64"])
@pytest.mark.parametrize("D,variant", [(2, "6"), (2, "7"), (3, "3")])
def test_two_faces_per_thread(monkeypatch, D, variant, precision):
    want = one_step(monkeypatch, D, "0", precision)
    got = one_step(monkeypatch, D, variant, precision)
    assert np.isfinite(want).all() and np.isfinite(got).all()
    # single-precision sums of a face in another order: 40 roundings of 2^-24 of the variable's largest value
    assert np.all(np.abs(got - want) < 40 * 2.0 ** -24 * (np.abs(want).max(1, keepdims=True) + 1e-17))


@pytest.mark.parametrize("D,expand", [(1, "directional"), (2, "directional"), (2, "multid"), (3, "multid")])
def test_fp64_face(D, expand):
    torch = pytest.importorskip("torch")
    z = np.linspace(15.642, 15.68, 20)
    u, p = z * np.sqrt(2.0 / 1.4), 1 / 1.4
    nv = D + 2

    def side(sign):
        U = np.zeros((z.size, D))
        U[:, 0] = sign * u
        return 1e-200 * np.concatenate([np.ones((z.size, 1)), U, (p / 0.4 + 0.5 * (U * U).sum(1))[:, None]], 1)

    wl, wr = side(-1), side(1)
    zero = np.zeros((z.size, (2 + 2 * (D - 1)) * nv))
    rec = np.concatenate([wl, wr, wl, wr, zero, np.full((z.size, 2), 0.5), np.zeros((z.size, 1))], 1)
    F, _ = gks.face_flux(D, torch.tensor(rec, device="cuda"), 1e-2, mu=0.0, precision="fp64", expand=expand)
    F = F.cpu().numpy()
    assert np.isfinite(F).all()
    # at most dt |u| times the difference of the cells' energies goes through
    assert np.abs(F).max() <= 1e-2 * u.max() * 2 * np.abs(wl).max()
