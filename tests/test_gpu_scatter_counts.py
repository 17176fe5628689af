"""The key scatter's bands of tile rows follow the keys there are, not the room
for them: lists of one to six bands (one for every 13 MB of keys), with the
capacity just enough, many times the count, and too small, on grids of few
rows and of more tiles than a band's shared memory holds.  The lists are those
of the separate projection and binning calls, bit for bit."""
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev

pytestmark = pytest.mark.gpu

BAND_KEYS = (13 << 20) // 8


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


# (size, growth of the log-scales, bands the keys make)
@pytest.mark.parametrize("W,H,grow,bands", [
    (640, 480, 0.0, 1), (640, 480, 2.5, 2), (640, 480, 3.0, 3), (640, 480, 4.0, 6), (1920, 40, 4.0, 3), (1918, 1079, 2.2, 5),
    (1918, 1079, 0.0, 1)])
def test_bands_follow_the_count(G, W, H, grow, bands):
    n = 20011
    sc = S.surface_scene(n, 78)
    sc["log_scales"] += grow
    g = dev(sc)
    cs, cfg = G.camera(S.camera(W, H, 525.0 * W / 640.0)), G.default_config()
    rec = torch.empty((n, 12), device="cuda")
    proj = G.gs_project(cfg, cs, g)
    k = int(G.gs_bin_count(cs, proj, n, cfg=cfg).item())
    assert min(-(-k // BAND_KEYS), 6) == bands
    b = G.gs_bin_sort(cs, proj, n, k, cfg=cfg)
    for cap in (k, 8 * k + (8 << 20)):
        a = G.gs_project_bin_sort(cfg, cs, g, rec, cap)
        assert int(a[2].item()) == k
        assert torch.equal(a[0][:k], b[0][:k]) and torch.equal(a[1][:k], b[1][:k])
        assert torch.equal(a[3], b[3]) and torch.equal(a[4], b[4])
    # too small: the true count, ranges clipped to the capacity, every list an ordered part of the full one
    cap = k // 3
    a = G.gs_project_bin_sort(cfg, cs, g, rec, cap)
    assert int(a[2].item()) == k and G.gs_status_poll(blocking=True)[0] == G.GS_ERR_CAPACITY
    G.gs_status_reset()
    start, end = (b[3][:, i].long().clamp(max=cap) for i in (0, 1))
    held = end > start
    assert torch.equal(a[3][held].long(), torch.stack([start, end], 1)[held]) and int(a[3].max()) == cap
    full = held & (b[3][:, 1].long() <= cap)
    last = int(b[3][full][:, 1].max())  # tiles that fit whole: the same lists
    assert torch.equal(a[0][:last], b[0][:last]) and torch.equal(a[1][:last], b[1][:last])
    d = a[0][:cap]
    assert bool((d[1:] >= d[:-1]).all())
