"""The FP64 even form (a generated A with the edge row and column, by cosine and
sine transforms) against the general FP64 form, which the same A takes when the
caller supplies it.

Bar: 1e-12 of the maximum over every transfer, as for the FP64 form against the
oracle: both sum the same products through transforms of at most 2^24 points
with relative rounding 1.1e-16 a step.
"""
import numpy as np
import pytest

import oracle
from paper_1208_3210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def lh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3210_gb300 import build, lindhard
    build.build()
    return lindhard


def _both(lh, grid, band):
    import torch
    b = dict(band)
    if b.get("kind", 0) == 0:
        b["mu"] = oracle.solve_mu(0, b["t"], b["tp"], b["tpp"], b["gamma"], grid["npz"], b["filling"])
        b["filling"] = float("nan")
    A = torch.from_numpy(oracle.spectral(b, grid).astype(np.float64)).cuda().contiguous()
    plan = lh.Plan([grid], precision=lh.FP64)
    a = plan.imchi([b])
    g = plan.imchi([b], A_in=A)
    plan.status()
    plan.close()
    torch.cuda.synchronize()
    return a, g


# cosine lengths 16, 24, 32, 48, 64, 96, 128; lags from one to all of them
@pytest.mark.parametrize("zones,npz,q", [(2, 2, 2), (2, 2, 8), (3, 6, 30), (2, 10, 40), (2, 16, 64), (3, 16, 48),
                                         (2, 24, 96), (2, 32, 64), (5, 8, 60), (2, 48, 96), (3, 32, 160), (2, 64, 256),
                                         (4, 32, 200), (2, 84, 168)])
@pytest.mark.parametrize("ff_a", [0.0, 1.0])
def test_lengths(lh, zones, npz, q, ff_a):
    grid = wl.grid_params(zones, npz, 22, 2.0, q_extent=q)
    a, g = _both(lh, grid, wl.band_params(filling=1.1, gamma=0.08, ff_a=ff_a))
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())


# energy lengths 16 to 256, odd counts, few and all transfers
@pytest.mark.parametrize("n_eps,n_omega", [(2, 1), (3, 2), (16, 1), (23, 23), (37, 11), (48, 24), (64, 64), (90, 7),
                                           (128, 64), (129, 129), (192, 96), (256, 128)])
@pytest.mark.parametrize("quantity", [0, 1, 2])
def test_energies(lh, n_eps, n_omega, quantity):
    if quantity and n_eps + n_omega - 1 > 256:
        pytest.skip("beyond the FP64 energy lengths")
    grid = wl.grid_params(2, 6, n_eps, 2.0, n_omega=n_omega, quantity=quantity, q_extent=20)
    band = wl.band_params(filling=1.1, gamma=0.08, ff_a=0.5, **({"kT": 0.06} if quantity else {}))
    a, g = _both(lh, grid, band)
    # the rounding of the energy transforms spreads over all transfers, and the
    # kept ones may vanish (Im chi(q, 0) = 0)
    every = n_eps if not quantity else min(n_eps, 257 - n_eps)
    scale = g if n_omega >= every else _both(lh, dict(grid, n_omega=every), band)[1]
    assert float((a - g).abs().max()) <= TOL * float(scale.abs().max())


def test_free_electrons(lh):
    grid = wl.grid_params(2, 16, 40, 2.0)
    a, g = _both(lh, grid, wl.band_params(kind=1, mu=0.7, filling=float("nan"), gamma=0.1, ff_a=0.3))
    assert float((a - g).abs().max()) <= TOL * float(g.abs().max())
