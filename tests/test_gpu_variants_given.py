"""Every engine variant of the general form against the FP64 oracle, each pinned
through a tune-cache file, with the spectral function supplied by the caller: a
generated one on several zones takes the even form and none of these passes.

The p_y passes, the product pass and the inverse energy pass of one-third padding
(P = 192, 384, 1536), of a power of two (one zone, P = 128), at every energy
length of the warp-per-line passes, and at finite temperature.  Bar: 2e-5 of the
maximum (FP32), on seeded samples; random spectral functions without symmetry.
"""
import json

import numpy as np
import pytest

import oracle
from paper_1208_3210_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL32 = 2e-5
# as the autotuner's lists: 12-value tiles at 3 * 2^k lengths, wide tiles from
# 384 on, the pruned engine (6-10) where the padding is a third
PY = {"pow2": [0, 1, 3, 5], "third": [0, 1, 2, 3, 4, 5, 8, 9], "long": [0, 1, 2, 3, 4, 5, 6, 8, 9, 10, 11]}
PX = {"pow2": [0, 2, 4], "third": [0, 1, 2, 3, 4, 6, 7], "long": [0, 1, 2, 3, 4, 5, 6, 7, 8, 9, 10]}


@pytest.fixture(scope="module")
def lh():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_3210_gb300 import build, lindhard
    build.build()
    return lindhard


class Pinned:
    """Plans of one grid with chosen variants, and the oracle's samples."""

    def __init__(self, lh, grid, tmp_path, monkeypatch, kT=0.0, count=150, A=None):
        import torch
        self.lh, self.grid, self.tmp, self.mp = lh, grid, tmp_path, monkeypatch
        self.kT, self.quantity = kT, grid.get("quantity", 0)
        A = wl.random_spectral(grid, seed=17) if A is None else A
        self.A = torch.from_numpy(A).cuda().reshape(-1)
        self.lx, self.ly, self.m = wl.output_samples(grid, count, seed=3, near_origin=4)
        A64, Q = A.astype(np.float64), grid["q_extent"]
        self.ref = (oracle.thermal_samples(A64, grid, Q, kT, self.quantity, self.lx, self.ly, self.m)
                    if self.quantity else oracle.imchi_samples(A64, grid, Q, self.lx, self.ly, self.m))
        probe = lh.Plan([grid])
        s = self.sizes = probe.sizes[0]
        probe.close()
        self.key = f"{torch.cuda.get_device_name(0)}|P={s.fft_p}|N={s.N}|PE={s.fft_e}|Q={s.q_extent}|"

    def error(self, fwd=1, inv=1, px=0, ve=0):
        import torch
        path = self.tmp / f"tune_{fwd}_{inv}_{px}_{ve}.json"
        path.write_text(json.dumps({self.key + "fwd_y": fwd, self.key + "inv_y": inv, self.key + "x_product": px,
                                    self.key + "inv_energy": ve}, indent=0))
        self.mp.setenv("LINDHARD_TUNE_CACHE", str(path))
        plan = self.lh.Plan([self.grid], autotune=True)
        assert plan.variants() == {"py_fwd": fwd, "py_inv": inv, "px_product": px, "energy_inv": ve}
        out = plan.imchi([wl.band_params(kT=self.kT)] if self.quantity else None, A_in=self.A)
        plan.status()
        plan.close()
        s = self.sizes
        idx = [torch.from_numpy(a.astype(np.int64)).cuda() for a in (self.lx, self.ly, self.m)]
        got = out.reshape(s.q_extent, s.q_extent, s.n_omega)[idx[0], idx[1], idx[2]].double().cpu().numpy()
        return np.abs(got - self.ref).max() / np.abs(self.ref).max()

    def check_all(self, family, inverse_energy):
        for v in PY[family]:
            assert self.error(fwd=v) <= TOL32, ("fwd_y", v)
            assert self.error(inv=v) <= TOL32, ("inv_y", v)
        for v in PX[family]:
            assert self.error(px=v) <= TOL32, ("x_product", v)
        for v in inverse_energy:
            assert self.error(ve=v) <= TOL32, ("inv_energy", v)


@pytest.mark.parametrize("grid,family,p", [
    (wl.grid_params(2, 64, 40, 1.5), "third", 192), (wl.grid_params(1, 128, 32, 1.0), "pow2", 128),
    (wl.grid_params(4, 64, 128, 2.0), "long", 384)], ids=["P192", "P128_one_zone", "P384"])
def test_every_variant(lh, grid, family, p, tmp_path, monkeypatch):
    pin = Pinned(lh, grid, tmp_path, monkeypatch)
    assert pin.sizes.fft_p == p
    pin.check_all(family, [0, 1, 2] if grid["n_eps"] >= 128 else [0, 1])


@pytest.mark.parametrize("quantity", [1, 2])
def test_every_variant_at_finite_temperature(lh, quantity, tmp_path, monkeypatch):
    pin = Pinned(lh, wl.grid_params(2, 64, 24, 1.5, quantity=quantity), tmp_path, monkeypatch, kT=0.04)
    assert pin.sizes.fft_p == 192
    pin.check_all("third", [0, 1])


@pytest.mark.parametrize("n_eps,n_omega,quantity", [(128, 64, 0), (100, 50, 0), (256, 128, 0), (200, 200, 0), (512, 256, 0),
                                                    (333, 7, 0), (512, 512, 0), (256, 128, 1), (193, 192, 2), (512, 256, 2)])
def test_inverse_energy_variants(lh, n_eps, n_omega, quantity, tmp_path, monkeypatch):
    pin = Pinned(lh, wl.grid_params(2, 48, n_eps, 2.0, n_omega=n_omega, quantity=quantity), tmp_path, monkeypatch,
                 kT=0.05 if quantity else 0.0, count=100)
    assert pin.sizes.fft_e in (128, 256, 384, 512, 768) and pin.sizes.fft_p == 192
    for v in (0, 1, 2):
        assert pin.error(ve=v) <= TOL32, v


def test_every_variant_at_full_size(lh, tmp_path, monkeypatch):
    import torch
    grid = wl.WORKLOADS["large_1024x1024x512"]["grid"]
    # a random A (every cell drawn alike) has a large mean: the spectral function
    # of the band, off centre, keeps the samples' spread and has no symmetry
    band = dict(wl.WORKLOADS["large_1024x1024x512"]["band"])
    band["mu"] = oracle.solve_mu(0, band["t"], band["tp"], band["tpp"], band["gamma"], grid["npz"], band["filling"])
    A = oracle.spectral(band, grid).astype(np.float32)
    A = np.ascontiguousarray(np.roll(A, (37, -101), axis=(0, 1)))
    pin = Pinned(lh, grid, tmp_path, monkeypatch, count=150, A=A)
    del A
    assert pin.sizes.fft_p == 1536 and pin.sizes.fft_e == 512
    pin.check_all("long", [0, 1, 2])
    del pin
    torch.cuda.empty_cache()
