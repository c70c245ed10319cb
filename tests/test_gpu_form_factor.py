"""|M(p)|^2 = exp(-|p|^2 ff_a^2 / 8) for any finite ff_a: where ff_a^2 is beyond FP64
the weight is 1 at p = 0 and 0 elsewhere, as for any ff_a that long."""
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


@pytest.mark.parametrize("ff_a", [1e155, 1e300])
@pytest.mark.parametrize("zones", [1, 2])
def test_form_factor_of_any_length(lh, zones, ff_a):
    grid = wl.grid_params(zones, 16, 16, 1.0)
    band = wl.band_params(filling=float("nan"), mu=0.1, gamma=0.1, ff_a=ff_a)
    plan = lh.Plan([grid])
    a = plan.imchi([band])
    b = plan.imchi([dict(band, ff_a=1e100)])
    plan.status()
    plan.close()
    assert bool(a.isfinite().all()) and float((a - b).abs().max()) == 0.0
