"""The chemical potential solved in one CTA (zones of at most 160 points per
axis) against the oracle's FP64 bisection: class counts around a warp's and a
block's edges, narrow and wide Lorentzians, nearly empty and nearly full bands.

Bar: 1e-12 eV plus 4e-16 of the bracket.  The last step works on sums rounded at
2^-47 and is cubic from 1e-6 eV: (1e-6 / gamma)^2 1e-6 is 2.5e-13 eV at the
smallest gamma here.
"""
import math

import pytest

import oracle
from paper_1208_3210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3210_gb300 import build, lindhard
    build.build()
    return lindhard


def _solve(lh, npz, band):
    import torch
    plan = lh.Plan([wl.grid_params(2, npz, 4, 1.0, q_extent=2)])
    mu = torch.zeros(1, dtype=torch.float64, device="cuda")
    plan.imchi([band], mu_out=mu)
    plan.status()
    plan.close()
    return mu.item()


@pytest.mark.parametrize("npz", [4, 6, 20, 62, 64, 66, 126, 128, 158, 160, 162])
@pytest.mark.parametrize("gamma,filling", [(0.002, 1.15), (0.01, 0.7), (0.05, 1.04), (0.05, 1.0), (0.2, 1.6), (0.3, 0.45)])
def test_mu_against_bisection(lh, npz, gamma, filling):
    band = wl.band_params(filling=filling, gamma=gamma)
    ref = oracle.solve_mu(0, band["t"], band["tp"], band["tpp"], gamma, npz, filling)
    assert abs(_solve(lh, npz, band) - ref) <= 1e-12 + 4e-16 * 12


@pytest.mark.parametrize("npz,filling", [(16, 0.3), (64, 0.6), (160, 1.1)])
def test_mu_free_electrons(lh, npz, filling):
    band = wl.band_params(filling=filling, gamma=0.05, kind=1, t=0.0, tp=0.0, tpp=0.0)
    ref = oracle.solve_mu(1, 0.0, 0.0, 0.0, 0.05, npz, filling)
    got = _solve(lh, npz, band)
    assert abs(got - ref) <= 1e-12 + 4e-16 * 25 and math.isfinite(got)
