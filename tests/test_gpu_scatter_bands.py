"""The key scatter in bands of tile rows (large key capacities) and with
Gaussians of very different tile counts in one warp: the lists are those of
the separate projection and binning calls, bit for bit."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


# capacities of 1, 2, 3 and 6 bands; grids of few rows (fewer than the bands,
# a remainder in the last band) and strides
@pytest.mark.parametrize("cap", [200_000, 2_700_000, 6_000_000, 40_000_000])
@pytest.mark.parametrize("W,H,sx,sy", [(640, 480, 1, 1), (333, 41, 1, 1), (320, 16, 1, 1), (1200, 680, 2, 4)])
def test_banded_scatter_equals_the_two_calls(G, cap, W, H, sx, sy):
    n = 9001
    sc = S.surface_scene(n, 77)
    sc["log_scales"][::50] += 3.0   # some Gaussians cover most of the grid
    g = dev(sc)
    cam = S.camera(W, H, 525.0 * W / 640.0, sx=sx, sy=sy)
    cs, cfg = G.camera(cam), G.default_config()
    rec = torch.empty((n, 12), device="cuda")
    a = G.gs_project_bin_sort(cfg, cs, g, rec, cap)
    b = G.gs_bin_sort(cs, G.gs_project(cfg, cs, g), n, cap, cfg=cfg)
    k = int(a[2].item())
    assert 0 < k <= cap and k == int(b[2].item())
    assert torch.equal(a[0][:k], b[0][:k]) and torch.equal(a[1][:k], b[1][:k])
    assert torch.equal(a[3], b[3]) and torch.equal(a[4], b[4])
    assert np.all(np.diff(a[0][:k].cpu().numpy().view(np.uint64).astype(np.float64)) >= 0)
