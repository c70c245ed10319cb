"""Which bands may leave out the zone edge in the even form (ev_band_applies).

Free electrons are not periodic: with mu near the edge's energy the edge row
lies on the Fermi level while the heavier rows near the centre carry only
Lorentzian tails, so there the form factor alone says nothing.  Im chi is held to
the FP32 bar of 2e-5 of its maximum against the FP64 oracle, the parameter
gradient to 1e-6 max|dL/dA| sum|dA/dtheta| of the general form, which the call
takes when dL/dA is asked for too (both as in test_gpu_even.py).  Tight-binding
bands are checked on both sides of the rule for an even and an odd count of
zones, at mu in the band and at its top, where only the zone's corners are left.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1208_3210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL32 = 2e-5
NAN = float("nan")


@pytest.fixture(scope="module")
def lh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3210_gb300 import build, lindhard
    build.build()
    return lindhard


def _error(lh, grid, band):
    plan = lh.Plan([grid])
    out = plan.imchi([band])
    plan.status()
    plan.close()
    Q, n = grid["q_extent"], grid["n_omega"]
    ref = oracle.imchi_full(oracle.spectral(band, grid), grid, Q, n)
    return np.abs(out.cpu().numpy().astype(np.float64).reshape(Q, Q, n) - ref).max() / np.abs(ref).max()


# (zones pi)^2 / 2 = 78.96 and 123.37: the edge's energy; ff_a just above
# (zones pi ff_a)^2 / 8 = 24 ln 2 (0.918 and 0.735) and well above
FREE = [(4, 0.92, 79.0, 0.05, 32), (4, 1.0, 79.0, 0.05, 32), (4, 0.92, 85.0, 0.05, 32), (4, 0.92, 79.0, 0.005, 128),
        (5, 0.75, 123.4, 0.05, 32), (4, 0.92, 0.7, 0.05, 32), (4, 0.92, 40.0, 0.05, 32)]


@pytest.mark.parametrize("zones,ff_a,mu,gamma,n_eps", FREE)
def test_free_electrons_near_the_edge_energy(lh, zones, ff_a, mu, gamma, n_eps):
    grid = wl.grid_params(zones, 12, n_eps, 1.0, n_omega=min(n_eps // 2, 24))
    band = wl.band_params(kind=1, mu=mu, filling=NAN, gamma=gamma, ff_a=ff_a)
    assert _error(lh, grid, band) <= TOL32


@pytest.mark.parametrize("zones,ff_a,mu,gamma,n_eps", FREE)
def test_free_electron_gradient_near_the_edge_energy(lh, zones, ff_a, mu, gamma, n_eps):
    import torch
    grid = wl.grid_params(zones, 12, n_eps, 1.0)
    band = wl.band_params(kind=1, mu=mu, filling=NAN, gamma=gamma, ff_a=ff_a)
    w = torch.from_numpy(wl.loss_weights(grid, seed=3)).cuda().reshape(-1)
    plan = lh.Plan([grid], backward=True)
    dp, ref = (torch.zeros(5, dtype=torch.float64, device="cuda") for _ in range(2))
    dA = torch.empty(plan.a_elems(), device="cuda")
    plan.backward(w, bands=[band], dparams=dp)
    plan.backward(w, bands=[band], dA=dA, dparams=ref)
    plan.status()
    plan.close()
    scale = float(dA.abs().max()) * np.abs(oracle.spectral_dtheta(band, grid)).reshape(5, -1).sum(1)
    assert np.all(np.abs((dp - ref).cpu().numpy())[3:] <= 1e-6 * scale[3:])


# (zones pi ff_a)^2 - [zones odd] (pi ff_a)^2 = 192 ln 2 at 0.918 (4 zones) and 1.298 (3)
@pytest.mark.parametrize("zones,ff_a", [(4, 0.91), (4, 0.93), (3, 1.23), (3, 1.29), (3, 1.31), (2, 1.83), (2, 1.85)])
@pytest.mark.parametrize("mu", [0.0, 1.81])
def test_tight_binding_on_both_sides(lh, zones, ff_a, mu):
    grid = wl.grid_params(zones, 12, 32, 0.5)
    assert _error(lh, grid, wl.band_params(filling=NAN, mu=mu, gamma=0.02, ff_a=ff_a)) <= TOL32


def test_gradient_of_a_batch_on_both_routes(lh):
    """One call whose instances take the even form, the general one (the edge
    carried) and free electrons: each as alone."""
    import torch
    grid = wl.grid_params(4, 12, 40, 1.5)
    bands = [wl.band_params(filling=1.1, gamma=0.1, ff_a=f) for f in (0.93, 0.91, 0.0)]
    bands.append(wl.band_params(kind=1, mu=79.0, filling=NAN, gamma=0.1, ff_a=0.93))
    n = len(bands)
    w1 = torch.from_numpy(wl.loss_weights(grid, seed=5)).cuda().reshape(-1)
    dp = torch.zeros(n, 5, dtype=torch.float64, device="cuda")
    for concurrent in (False, True):
        plan = lh.Plan([grid] * n, backward=True, concurrent=concurrent)
        plan.backward(w1.repeat(n), bands=bands, dparams=dp)
        plan.status()
        plan.close()
        for i, b in enumerate(bands):
            one = torch.zeros(5, dtype=torch.float64, device="cuda")
            alone = lh.Plan([grid], backward=True)
            alone.backward(w1, bands=[b], dparams=one)
            alone.status()
            alone.close()
            assert torch.equal(dp[i], one) and math.isfinite(float(one.abs().sum()))
