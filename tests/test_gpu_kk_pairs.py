"""Lines of the Kramers-Kronig pass share transforms; what one line holds stays
out of its neighbour's result, whatever the ratio of the two.

Bar: 1e-6 of the line's own maximum, as in test_gpu_kk.py for one scale.
"""
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


def _plan(lh, n):
    return lh.Plan([wl.grid_params(2, 6, max(2, n), 1.5, n_omega=n)])


# scales of consecutive lines; 2^126 makes sums inside a transform overflow
@pytest.mark.parametrize("n", [30, 64, 100, 128, 190, 256])
@pytest.mark.parametrize("scales", [(1.0, 1e-4), (1e-8, 1.0), (1.0, 1e-30), (2.0 ** 126, 1.0), (1e-20, 1e-36), (1.0, 0.0)])
def test_lines_of_different_scale(lh, n, scales):
    import torch
    plan = _plan(lh, n)
    g = torch.Generator().manual_seed(n)
    im = -torch.rand(144, n, generator=g)
    im *= torch.tensor(scales).repeat(72)[:, None]
    re, _ = plan.kk_rpa(im.cuda().reshape(-1), rpa=False, variant=0)
    plan.status()
    plan.close()
    x = im.numpy().astype(np.float64)
    ref = oracle.kk_real(x.reshape(12, 12, n)).reshape(144, n)
    got = re.cpu().numpy().astype(np.float64).reshape(144, n)
    bar = 1e-6 * np.maximum(np.abs(ref).max(1), np.abs(x).max(1))
    ok = np.abs(ref).max(1) < 3e38
    assert np.all(np.abs(got - ref).max(1)[ok] <= bar[ok] + 1e-44)
