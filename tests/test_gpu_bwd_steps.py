"""The masked backward's steps of four entries (sums over a warp's pixels on
the tensor cores) at the list lengths where they can go wrong: padded last
steps, runs that end inside a step, the ring's wrap at 64 entries, and warps
whose block sees few or none of the entries."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev, np_of, pack_splats, rel_l2

pytestmark = pytest.mark.gpu

# both paths sum float32 terms of one sign pattern; the split keeps 23 of a
# term's 24 bits, so a field differs from the float32 path by its own rounding
# (up to ~100 terms per sum): below 1e-5 relative in norm
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
@pytest.mark.parametrize("sx,sy", [(1, 1), (2, 2), (4, 1), (1, 4), (1, 2), (2, 1)])
@pytest.mark.parametrize("mode", ["track", "map"])
def test_masked_backward_equals_unmasked_at_step_edges(G, n, sx, sy, mode):
    W, H = 30 * sx, 21 * sy
    cam = S.camera(W, H, 100.0, sx=sx, sy=sy)
    # wide faint Gaussians on every block, every fifth one small
    s = S.splats(n, W, H, seed=900 + n, sigma_px=(8.0 * max(sx, sy), 14.0 * max(sx, sy)), opaque_frac=0.0, cull_frac=0.0)
    s["opacity"] *= 0.06
    s["opacity"] += 0.02
    small = np.arange(n) % 5 == 4
    s["conic"][small] = np.array([0.8, 0.1, 0.6], np.float32)
    s["radius"][small] = 4
    rec = pack_splats(s)
    cfg, cs = G.default_config(), G.camera(cam)
    cap = 64 * n + 64
    _, vals, nk, ranges, order = G.gs_bin_sort(cs, rec, n, cap)
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    out = G.gs_render_fwd(cfg, cs, rec, n, vals, ranges, order=order, masks=bm)
    Ws, Hs, _, _ = G.grid(cam)
    d_rgb, d_dep = (torch.from_numpy(x).cuda() for x in S.image_grads(Ws, Hs, n))
    z = dev({"means": np.zeros((n, 3), np.float32), "log_scales": np.zeros((n, 3), np.float32),
             "quats": np.zeros((n, 4), np.float32), "opacity_logit": np.zeros(n, np.float32),
             "rgb": np.zeros((n, 3), np.float32)})
    g2 = [np_of(G.gs_render_bwd(cfg, cs, z, rec, vals, ranges, out["t_final"], out["last_idx"], d_rgb, d_dep,
                                mode=G.GS_MAP if mode == "map" else G.GS_TRACK, order=order, masks=k))
          for k in (None, bm)]
    assert int(nk.item()) <= cap and np.any(g2[0])
    for cols in ([0, 1], [2, 3, 4], [5], [6], [8, 9, 10]):
        if mode == "track" and cols in ([5], [8, 9, 10]):
            assert not g2[1][:, cols].any()
        else:
            assert rel_l2(g2[1][:, cols], g2[0][:, cols]) <= TOL, (cols, rel_l2(g2[1][:, cols], g2[0][:, cols]))
