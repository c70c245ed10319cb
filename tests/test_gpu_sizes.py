"""lindhard_plan_sizes: the bytes and launches of a call with A generated are
those of the form that the call takes (every intermediate written once and read
once, its non-redundant entries only)."""
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


def _sizes(lh, grid, **kw):
    plan = lh.Plan([grid], **kw)
    s = plan.sizes[0]
    plan.close()
    return s


@pytest.mark.parametrize("grid,M,ne", [
    (wl.grid_params(4, 64, 256, 2.0), 192, 256), (wl.grid_params(8, 128, 512, 3.0), 768, 512),
    (wl.grid_params(5, 36, 150, 2.0, quantity=2), 144, 150), (wl.grid_params(3, 50, 201, 2.0, n_omega=30, q_extent=300), 192, 60)])
def test_even_form(lh, grid, M, ne):
    s = _sizes(lh, grid)
    tri = M * (M + 1) // 2
    B = s.N // 2 * M * ne + tri * (ne + s.n_omega) + (s.q_extent // 2 + 1) * M * s.n_omega
    assert s.hbm_bytes_forward == 4 * (2 * B + s.out_elems)
    assert s.kernels_forward == 6


def test_even_form_in_double_precision(lh):
    grid = wl.grid_params(2, 32, 128, 2.0)
    s = _sizes(lh, grid, precision=lh.FP64)
    M, ne, n = 48, 128, 64
    B = 33 * M * ne + M * (M + 1) // 2 * (ne + 4 * n) + 2 * s.q_extent * M * n
    assert s.hbm_bytes_forward == 8 * (2 * B + s.out_elems)
    assert s.kernels_forward == 7   # the edge's lines are always formed


@pytest.mark.parametrize("grid,kw", [(wl.grid_params(1, 32, 48, 1.0), {}), (wl.grid_params(2, 64, 128, 2.0), dict(persistent=True)),
                                     (wl.grid_params(1, 32, 48, 1.0), dict(precision=2))])
def test_general_form(lh, grid, kw):
    s = _sizes(lh, grid, **kw)
    H, cb = s.fft_e // 2 + 1, 16 if kw.get("precision") == 2 else 8
    W = s.N * s.N * 2 * H + s.N * s.fft_p * 2 * H + s.q_extent * s.fft_p * H + s.q_extent ** 2 * H
    assert s.hbm_bytes_forward == 2 * W * cb + s.out_elems * cb // 2
    assert s.kernels_forward == (1 if kw.get("persistent") else 6)
