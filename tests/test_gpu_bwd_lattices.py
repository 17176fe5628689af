"""The masked backward's one-warp CTAs on the small tiles of strided frames, at
the list lengths where its steps of four entries, its runs of 32 and its ring
of 64 can go wrong.  The grids have enough tiles for that kernel (1024 of 64
pixels, 2048 of 32, 4096 of 16); the Gaussians lie in one corner of them."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev, np_of, pack_splats, rel_l2

pytestmark = pytest.mark.gpu

# two float32 summation orders of the same terms (tests/test_gpu_parity.py's bound for it)
TOL = 1e-5


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 67, 130, 257])
@pytest.mark.parametrize("sx,sy", [(2, 2), (4, 1), (1, 4), (4, 2), (2, 4), (4, 4)])
@pytest.mark.parametrize("mode", ["track", "map"])
def test_small_tiles_at_step_edges(G, n, sx, sy, mode):
    W, H = 256 * sx - (sx > 1), 256 * sy - (sy > 1)
    cam = S.camera(W, H, 100.0, sx=sx, sy=sy)
    s = S.splats(n, 30 * sx, 21 * sy, seed=700 + n, sigma_px=(8.0 * max(sx, sy), 14.0 * max(sx, sy)), opaque_frac=0.0,
                 cull_frac=0.0)
    s["opacity"] = (0.02 + 0.06 * s["opacity"]).astype(np.float32)
    small = np.arange(n) % 3 == 2  # a few blocks see only some of the entries
    s["conic"][small] = np.array([0.8, 0.1, 0.6], np.float32)
    s["radius"][small] = 4
    rec, cs, cfg = pack_splats(s), G.camera(cam), G.default_config()
    cap = int(G.gs_bin_count(cs, rec, n, cfg=cfg).item())
    _, vals, _, ranges, order = G.gs_bin_sort(cs, rec, n, cap)
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    out = G.gs_render_fwd(cfg, cs, rec, n, vals, ranges, order=order, masks=bm)
    Ws, Hs, TX, TY = G.grid(cam)
    assert TX * TY >= {64: 1024, 32: 2048, 16: 4096}[(256 // TX) * (256 // TY)]
    d_rgb, d_dep = (torch.from_numpy(x).cuda() for x in S.image_grads(Ws, Hs, n))
    z = dev({"means": np.zeros((n, 3), np.float32), "log_scales": np.zeros((n, 3), np.float32),
             "quats": np.zeros((n, 4), np.float32), "opacity_logit": np.zeros(n, np.float32),
             "rgb": np.zeros((n, 3), np.float32)})
    g2 = [np_of(G.gs_render_bwd(cfg, cs, z, rec, vals, ranges, out["t_final"], out["last_idx"], d_rgb, d_dep,
                                mode=G.GS_MAP if mode == "map" else G.GS_TRACK, order=order, masks=k))
          for k in (None, bm)]
    assert np.any(g2[0])
    for cols in ([0, 1], [2, 3, 4], [5], [6], [8, 9, 10]):
        if mode == "track" and cols in ([5], [8, 9, 10]):
            assert not g2[1][:, cols].any()
        else:
            assert rel_l2(g2[1][:, cols], g2[0][:, cols]) <= TOL, (cols, rel_l2(g2[1][:, cols], g2[0][:, cols]))


@pytest.mark.parametrize("n", [7199, 7200])
def test_either_side_of_the_line_between_the_kernels(G, n):
    """300 tiles of 64 pixels: with 24 Gaussians a tile the entry-parallel
    kernel takes over from the one-warp CTAs."""
    W, H = 320, 240
    cam = S.camera(W, H, 100.0, sx=2, sy=2)
    s = S.splats(n, W, H, seed=n, opaque_frac=0.02)
    rec, cs, cfg = pack_splats(s), G.camera(cam), G.default_config()
    cap = int(G.gs_bin_count(cs, rec, n, cfg=cfg).item())
    _, vals, _, ranges, order = G.gs_bin_sort(cs, rec, n, cap)
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    out = G.gs_render_fwd(cfg, cs, rec, n, vals, ranges, order=order, masks=bm)
    d_rgb, d_dep = (torch.from_numpy(x).cuda() for x in S.image_grads(W // 2, H // 2, n))
    z = dev({"means": np.zeros((n, 3), np.float32), "log_scales": np.zeros((n, 3), np.float32),
             "quats": np.zeros((n, 4), np.float32), "opacity_logit": np.zeros(n, np.float32),
             "rgb": np.zeros((n, 3), np.float32)})
    g2 = [np_of(G.gs_render_bwd(cfg, cs, z, rec, vals, ranges, out["t_final"], out["last_idx"], d_rgb, d_dep,
                                mode=G.GS_MAP, order=order, masks=k)) for k in (None, bm)]
    for cols in ([0, 1], [2, 3, 4], [5], [6], [8, 9, 10]):
        assert rel_l2(g2[1][:, cols], g2[0][:, cols]) <= TOL, (cols, rel_l2(g2[1][:, cols], g2[0][:, cols]))
