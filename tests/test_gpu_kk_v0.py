"""chi_RPA = chi / (1 - V_q chi), V_q = v0 / |q|^2, for v0 far from 1: one so small
that v0 / dp^2 leaves FP32's range still takes chi_RPA to its limit 0 at q = 0,
and one near or beyond FP32's largest gives what the form that divides in FP64
(variant 1) gives.

Bar: 2e-6 of the largest |chi_RPA| or |chi|: both forms carry Re chi to 1e-6.
"""
import pytest

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


@pytest.mark.parametrize("v0", [1e-50, -1e-300, 1e-40, 1e38, -1e38, 1e45])
def test_interactions_beyond_fp32(lh, v0):
    import torch
    plan = lh.Plan([wl.grid_params(2, 6, 32, 1.5, n_omega=32)])
    g = torch.Generator(device="cuda").manual_seed(3)
    im = -torch.rand(plan.out_elems(), generator=g, device="cuda")
    re0, rp0 = plan.kk_rpa(im, v0=v0, variant=0)
    re1, rp1 = plan.kk_rpa(im, v0=v0, variant=1)
    plan.status()
    plan.close()
    assert float(rp0[6, 6].abs().max()) == 0.0 and float(rp1[6, 6].abs().max()) == 0.0
    a, b = torch.view_as_real(rp0), torch.view_as_real(rp1)
    assert torch.equal(a.isnan(), b.isnan())
    assert float((a - b).nan_to_num(0.0).abs().max()) <= 2e-6 * float(b.nan_to_num(0.0).abs().max() + re1.abs().max())
