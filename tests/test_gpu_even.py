"""The even form of the forward call (a generated A is even in p_x and p_y and
symmetric under their exchange: cosine transforms of one quadrant) against the
general form, which the same A takes when the caller supplies it, and against
the FP64 oracle.

Bar: 2e-6 of the maximum between the two FP32 forms.  Each sums the same
products through transforms of log2 of at most 2^27 points with relative
rounding 6e-8 a step, about 3e-7 of the maximum each (their measured errors
against FP64), so 2e-6 leaves a factor of three for the maximum over all
outputs.
"""
import numpy as np
import pytest

import oracle
from paper_1208_3210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 2e-6


@pytest.fixture(scope="module")
def lh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3210_gb300 import build, lindhard
    build.build()
    return lindhard


def _both(lh, grid, band):
    """(generated A, the same A given) outputs of the grid's quantity."""
    import torch
    b = dict(band)
    if b.get("kind", 0) == 0:
        b["mu"] = oracle.solve_mu(0, b["t"], b["tp"], b["tpp"], b["gamma"], grid["npz"], b["filling"])
        b["filling"] = float("nan")
    A = torch.from_numpy(oracle.spectral(b, grid).astype(np.float32)).cuda().contiguous()
    plan = lh.Plan([grid])
    a = plan.imchi([b])
    g = plan.imchi([b], A_in=A)
    plan.status()
    plan.close()
    torch.cuda.synchronize()
    return a.double(), g.double()


# cosine lengths M: (N + Q/2)/2 rounded up to 16, 24, 32, ..., 2048
# in the order of the list: 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, ..., then
# the lengths 72, 144, 288, 432, 576, 864 and 1152
@pytest.mark.parametrize("zones,npz,q", [
    (4, 24, 92), (5, 36, 200), (4, 100, 340), (6, 96, 560), (8, 90, 820), (8, 150, 1000), (8, 192, 1400),
    (4, 4, 16), (5, 6, 30), (4, 10, 40), (4, 16, 64), (4, 20, 60), (5, 24, 118), (4, 32, 128), (6, 32, 2),
    (4, 64, 256), (4, 64, 512), (7, 50, 700), (8, 64, 512), (4, 160, 640), (8, 128, 1024), (8, 192, 2),
    (8, 240, 2000), (8, 256, 2048),
    (8, 256, 4096)])
def test_lengths(lh, zones, npz, q):
    big = zones * npz >= 1024
    grid = wl.grid_params(zones, npz, 6 if big else 34, 2.0, q_extent=q)
    a, g = _both(lh, grid, wl.band_params(filling=1.1, gamma=0.3 if big else 0.08, ff_a=1.4))
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())


# energy lengths 128, 256, 384, 512, 768; odd counts, few and all transfers
@pytest.mark.parametrize("n_eps,n_omega", [(2, 1), (3, 2), (16, 1), (37, 11), (128, 64), (129, 129), (200, 30),
                                           (256, 128), (300, 150), (384, 384), (401, 77), (512, 256), (700, 351),
                                           (768, 384)])
@pytest.mark.parametrize("quantity", [0, 1, 2])
def test_energies(lh, n_eps, n_omega, quantity):
    if quantity and n_eps + n_omega - 1 > 768:
        pytest.skip("beyond the even form's energy lengths")
    # The maximum is over every transfer: the rounding of the energy transforms
    # spreads over all of them, and the kept ones may vanish (Im chi(q, 0) = 0).
    grid = wl.grid_params(4, 12, n_eps, 2.0, n_omega=n_omega, quantity=quantity)
    band = wl.band_params(filling=1.1, gamma=0.08, ff_a=1.0, **({"kT": 0.06} if quantity else {}))
    a, g = _both(lh, grid, band)
    scale = float(_both(lh, dict(grid, n_omega=n_eps), band)[1].abs().max()) if n_omega < n_eps else float(g.abs().max())
    assert float((a - g).abs().max()) <= TOL * scale


def test_free_electrons(lh):
    grid = wl.grid_params(4, 16, 40, 2.0)
    a, g = _both(lh, grid, wl.band_params(kind=1, mu=0.7, filling=float("nan"), gamma=0.1, ff_a=1.0))
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())


@pytest.mark.parametrize("ff_a", [0.0, 0.9, 0.92, 1.5])
def test_both_sides_of_the_edge_weight(lh, ff_a):
    # 4 zones: (4 pi ff_a)^2 / 8 = 24 ln 2 at ff_a = 0.918
    grid = wl.grid_params(4, 16, 32, 1.5)
    band = wl.band_params(filling=1.1, gamma=0.08, ff_a=ff_a)
    b = dict(band, mu=oracle.solve_mu(0, band["t"], band["tp"], band["tpp"], band["gamma"], 16, 1.1))
    plan = lh.Plan([grid])
    got = plan.imchi([band]).cpu().numpy().astype(np.float64).reshape(64, 64, 16)
    plan.status()
    plan.close()
    ref = oracle.imchi_full(oracle.spectral(b, grid), grid, 64, 16)
    assert np.abs(got - ref).max() <= TOL * np.abs(ref).max()


# The edge row carried (few zones, small ff_a): every cosine length, lags from
# one to all of them, energy lengths 128 to 512, transfers of every remainder.
@pytest.mark.parametrize("zones,npz,q", [
    (2, 4, 2), (2, 4, 16), (3, 10, 60), (2, 16, 32), (2, 24, 96), (3, 20, 30), (2, 48, 96), (3, 36, 216), (2, 64, 256),
    (3, 50, 300), (2, 100, 300), (2, 128, 256), (4, 100, 340), (2, 192, 768), (6, 96, 560), (4, 128, 1024),
    (8, 90, 820), (4, 192, 1536), (8, 150, 1000), (4, 256, 2048), (8, 192, 1400), (8, 192, 3072), (8, 256, 4096)])
def test_edge_lengths(lh, zones, npz, q):
    big = zones * npz >= 1024
    grid = wl.grid_params(zones, npz, 6 if big else 34, 2.0, q_extent=q)
    a, g = _both(lh, grid, wl.band_params(filling=1.1, gamma=0.3 if big else 0.08, ff_a=0.3))
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())


@pytest.mark.parametrize("n_eps,n_omega", [(2, 1), (3, 2), (16, 1), (37, 11), (128, 64), (129, 129), (200, 30),
                                           (256, 128), (300, 150), (384, 384), (401, 77), (512, 256), (512, 512)])
@pytest.mark.parametrize("quantity", [0, 1, 2])
def test_edge_energies(lh, n_eps, n_omega, quantity):
    if quantity and n_eps + n_omega - 1 > 512:
        pytest.skip("beyond the energy lengths that carry the edge")
    grid = wl.grid_params(2, 12, n_eps, 2.0, n_omega=n_omega, quantity=quantity, q_extent=40)
    band = wl.band_params(filling=1.1, gamma=0.08, ff_a=0.0, **({"kT": 0.06} if quantity else {}))
    a, g = _both(lh, grid, band)
    scale = float(_both(lh, dict(grid, n_omega=n_eps), band)[1].abs().max()) if n_omega < n_eps else float(g.abs().max())
    assert float((a - g).abs().max()) <= TOL * scale


@pytest.mark.parametrize("quantity", [0, 1])
def test_edge_free_electrons_unaligned(lh, quantity):
    import torch
    grid = wl.grid_params(2, 16, 40, 2.0, quantity=quantity)
    band = wl.band_params(kind=1, mu=0.7, filling=float("nan"), gamma=0.1, ff_a=0.2, kT=0.05 if quantity else 0.0)
    a, g = _both(lh, grid, band)
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())
    plan = lh.Plan([grid])
    ref = plan.imchi([band])
    buf = torch.zeros(plan.out_elems() + 1, device="cuda")
    plan.imchi([band], out=buf[1:])
    plan.status()
    assert torch.equal(buf[1:], ref)
    plan.close()


def test_unaligned_output(lh):
    import torch
    grid = wl.grid_params(4, 16, 32, 1.5)
    band = wl.band_params(filling=1.1, gamma=0.08, ff_a=1.0)
    plan = lh.Plan([grid])
    ref = plan.imchi([band])
    buf = torch.zeros(plan.out_elems() + 1, device="cuda")
    plan.imchi([band], out=buf[1:])
    plan.status()
    assert torch.equal(buf[1:], ref)
    plan.close()


# Adjoint: the parameter gradient alone takes the even form, with dL/dA asked
# for too the general one.  Both sum dL/dA dA/dtheta with dL/dA within 5e-7 of
# its maximum (the measured error of either form on every cell), so each
# component agrees within 1e-6 max|dL/dA| sum|dA/dtheta|.
@pytest.mark.parametrize("zones,npz,n_eps,n_omega,q,quantity", [
    (4, 4, 3, 2, 16, 0), (4, 10, 34, 17, 40, 0), (5, 24, 37, 30, 118, 0), (4, 32, 128, 64, 128, 0),
    (4, 16, 201, 90, 128, 0), (6, 32, 20, 10, 2, 0), (4, 16, 300, 150, 64, 0), (4, 12, 512, 256, 48, 0),
    (4, 20, 401, 33, 60, 0), (4, 12, 40, 25, 48, 1), (4, 12, 150, 75, 48, 2), (4, 12, 200, 150, 60, 1),
    (4, 12, 300, 200, 48, 2), (4, 24, 30, 15, 92, 0), (5, 36, 20, 10, 200, 0), (6, 96, 8, 4, 560, 0)])
def test_parameter_gradient(lh, zones, npz, n_eps, n_omega, q, quantity):
    import torch
    grid = wl.grid_params(zones, npz, n_eps, 2.0, n_omega=n_omega, q_extent=q, quantity=quantity)
    band = wl.band_params(filling=1.1, gamma=0.1, ff_a=1.1, **({"kT": 0.06} if quantity else {}))
    w = torch.from_numpy(wl.loss_weights(grid, seed=3)).cuda().reshape(-1) - 0.3
    plan = lh.Plan([grid], backward=True)
    dp = torch.zeros(5, dtype=torch.float64, device="cuda")
    ref = torch.zeros(5, dtype=torch.float64, device="cuda")
    dA = torch.empty(plan.a_elems(), device="cuda")
    plan.backward(w, bands=[band], dparams=dp)
    plan.backward(w, bands=[band], dA=dA, dparams=ref)
    plan.status()
    plan.close()
    b = dict(band, mu=oracle.solve_mu(0, band["t"], band["tp"], band["tpp"], band["gamma"], npz, 1.1))
    scale = float(dA.abs().max()) * np.abs(oracle.spectral_dtheta(b, grid)).reshape(5, -1).sum(1)
    assert np.all(np.abs((dp - ref).cpu().numpy()) <= 1e-6 * scale), ((dp - ref).cpu().numpy() / scale)


def test_parameter_gradient_free_electrons(lh):
    import torch
    grid = wl.grid_params(4, 16, 40, 2.0)
    band = wl.band_params(kind=1, mu=0.7, filling=float("nan"), gamma=0.1, ff_a=1.0)
    w = torch.from_numpy(wl.loss_weights(grid, seed=3)).cuda().reshape(-1)
    plan = lh.Plan([grid], backward=True)
    dp, ref = (torch.zeros(5, dtype=torch.float64, device="cuda") for _ in range(2))
    dA = torch.empty(plan.a_elems(), device="cuda")
    plan.backward(w, bands=[band], dparams=dp)
    plan.backward(w, bands=[band], dA=dA, dparams=ref)
    plan.status()
    plan.close()
    scale = float(dA.abs().max()) * np.abs(oracle.spectral_dtheta(band, grid)).reshape(5, -1).sum(1)
    assert dp[:3].abs().max().item() == 0.0
    assert np.all(np.abs((dp - ref).cpu().numpy())[3:] <= 1e-6 * scale[3:])
