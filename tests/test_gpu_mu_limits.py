"""The chemical potential at the limits of its solves, against a bisection on
exactly rounded sums (math.fsum; the oracle's own plain FP64 sum of 16384
occupations is off by 2e-10 of a state, 1e-10 eV where n(mu) is flat): Lorentzians
so narrow that a step's remainder (d / gamma)^2 d counts, fillings in the tails, where
n(mu) is nearly flat, and zones on either side of 160 points per axis (one CTA up
to there, several passes beyond).

Bars.  Narrow Lorentzians: the solve's last step is repeated until its length d
has d^3 <= 1e-13 gamma^2, and the remainder of such a step is d (d / gamma)^2
times a constant that is large only where mu lies between two levels; with up to
fifty of it, 5e-12 eV.  Tails: 1e-10 eV as in test_gpu_mu.py.
"""
import math

import numpy as np
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


def _solve(lh, npz, bands):
    import torch
    plan = lh.Plan([wl.grid_params(2, npz, 4, 1.0, q_extent=2)])
    mu = torch.zeros(1, dtype=torch.float64, device="cuda")
    out = []
    try:
        for b in bands:
            plan.imchi([b], mu_out=mu)
            plan.status()
            out.append(mu.item())
    finally:
        plan.close()
    return out


def _exact(band, npz):
    h = npz // 2
    a, b = np.triu_indices(h + 1)
    w = np.where((a == 0) | (a == h), 1.0, 2.0) * np.where((b == 0) | (b == h), 1.0, 2.0) * np.where(a == b, 1.0, 2.0)
    p = 2 * np.pi * np.arange(h + 1) / npz
    if band["kind"] == 1:
        e = 0.5 * (p[a] ** 2 + p[b] ** 2)
    else:
        c, c2 = np.cos(p), np.cos(2 * p)
        e = -2 * band["t"] * (c[a] + c[b]) - 4 * band["tp"] * c[a] * c[b] - 2 * band["tpp"] * (c2[a] + c2[b])
    target = band["filling"] * 0.5 * npz * npz
    mu = oracle.solve_mu(band["kind"], band["t"], band["tp"], band["tpp"], band["gamma"], npz, band["filling"])
    lo, hi = mu - 1e-6, mu + 1e-6
    for _ in range(36):
        mid = 0.5 * (lo + hi)
        n = math.fsum(w * (0.5 - np.arctan((e - mid) / band["gamma"]) / np.pi))
        lo, hi = (mid, hi) if n < target else (lo, mid)
    return 0.5 * (lo + hi)


@pytest.mark.parametrize("npz", [4, 32, 64, 98, 128, 160])
@pytest.mark.parametrize("gamma", [1e-5, 1e-4, 1e-3, 1.9e-3, 2e-3])
@pytest.mark.parametrize("kind", [0, 1])
def test_narrow_lorentzians(lh, npz, gamma, kind):
    hop = {} if kind == 0 else dict(kind=1, t=0.0, tp=0.0, tpp=0.0)
    bands = [wl.band_params(filling=f, gamma=gamma, **hop) for f in (0.2, 0.5, 0.9, 1.04, 1.15, 1.5, 1.8)]
    for b, got in zip(bands, _solve(lh, npz, bands)):
        assert abs(got - _exact(b, npz)) <= 5e-12, b["filling"]


@pytest.mark.parametrize("npz", [32, 64, 98, 128, 160])
@pytest.mark.parametrize("kind", [0, 1])
def test_fillings_in_the_tails(lh, npz, kind):
    hop = {} if kind == 0 else dict(kind=1, t=0.0, tp=0.0, tpp=0.0)
    B = 9.869604401089358 if kind else 4 * (0.42 + 0.10 + 0.065)
    bands = []
    for gamma in (0.002, 0.01, 0.03, 0.1):
        for f in (0.001, 0.003, 0.01, 1.9, 1.99, 1.997, 1.999):
            b = wl.band_params(filling=f, gamma=gamma, **hop)
            lo = oracle.filling(b["kind"], b["t"], b["tp"], b["tpp"], gamma, npz, -B - 2.9)
            hi = oracle.filling(b["kind"], b["t"], b["tp"], b["tpp"], gamma, npz, B + 2.9)
            if lo < f < hi:
                bands.append(b)
    assert len(bands) >= 14
    for b in bands:
        got, = _solve(lh, npz, [b])
        assert abs(got - _exact(b, npz)) <= 1e-10, (b["filling"], b["gamma"])


@pytest.mark.parametrize("npz", [160, 162, 256])
def test_unreachable_filling_on_both_sides_of_160(lh, npz):
    with pytest.raises(lh.LindhardError, match="ENOCONV"):
        _solve(lh, npz, [wl.band_params(filling=1.9999, gamma=0.2)])
    b = wl.band_params(filling=1.15, gamma=0.2)
    assert abs(_solve(lh, npz, [b])[0] - _exact(b, npz)) <= 1e-12
