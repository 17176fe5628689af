"""The forward's forms on grids of more than 2048 tiles.  The pixel-parallel
kernel has the same per-pixel arithmetic whatever the tiling, so its strided
renders are the full render's sampled pixels bit for bit, from one list entry
to several batches; the entry-parallel kernel's are to rounding.  The blend
masks of both feed the masked backward's one-warp CTAs."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev, np_of, pack_splats, rel_l2

pytestmark = pytest.mark.gpu

W, H = 752, 740  # 47 x 47 tiles: the strided grids are pixel-parallel too


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


def render(G, rec, n, sx, sy, cap):
    cs, cfg = G.camera(S.camera(W, H, 100.0, sx=sx, sy=sy)), G.default_config()
    _, vals, nk, ranges, order = G.gs_bin_sort(cs, rec, n, cap)
    assert int(nk.item()) <= cap
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    return cs, cfg, vals, ranges, order, bm, G.gs_render_fwd(cfg, cs, rec, n, vals, ranges, order=order, masks=bm)


@pytest.mark.parametrize("sx,sy", [(2, 2), (4, 2), (2, 4), (4, 4), (3, 3), (2, 1), (1, 2), (4, 1), (1, 4)])
@pytest.mark.parametrize("kind", ["sparse", "dense", "one_tile"])
def test_strided_forward_is_the_full_forward_sampled(G, kind, sx, sy):
    n = {"sparse": 700, "dense": 30_000, "one_tile": 1100}[kind]
    s = S.splats(n, W, H, seed=11 + n, opaque_frac=0.02)
    if kind == "one_tile":  # lists of more than a thousand faint entries around one corner of four tiles
        s["uv"] = (np.array([[320.0, 336.0]]) + np.random.default_rng(3).normal(0, 3.0, (n, 2))).astype(np.float32)
        s["opacity"] = (0.01 + 0.03 * s["opacity"]).astype(np.float32)
    rec, cap = pack_splats(s), 60 * n
    full = render(G, rec, n, 1, 1, cap)[-1]
    cs, cfg, vals, ranges, order, bm, out = render(G, rec, n, sx, sy, cap)
    for k in ("rgb", "depth", "t_final", "n_blended"):
        want = full[k][..., ::sy, ::sx].contiguous()
        if min(sx, sy) == 1 and max(sx, sy) == 2:  # tiles of 128 pixels
            assert torch.equal(out[k], want), k
        else:  # the same fragments unless T comes within rounding of t_eps (none here); other summation orders
            assert torch.allclose(out[k].float(), want.float(), rtol=0 if k == "n_blended" else 3e-5, atol=2e-5), k
    if kind == "one_tile":
        assert int(out["n_blended"].max()) > 200
    Ws, Hs, _, _ = G.grid(cs)
    d_rgb, d_dep = (torch.from_numpy(x).cuda() for x in S.image_grads(Ws, Hs, n))
    z = dev({"means": np.zeros((n, 3), np.float32), "log_scales": np.zeros((n, 3), np.float32),
             "quats": np.zeros((n, 4), np.float32), "opacity_logit": np.zeros(n, np.float32),
             "rgb": np.zeros((n, 3), np.float32)})
    g2 = [np_of(G.gs_render_bwd(cfg, cs, z, rec, vals, ranges, out["t_final"], out["last_idx"], d_rgb, d_dep,
                                mode=G.GS_MAP, order=order, masks=k)) for k in (None, bm)]
    for cols in ([0, 1], [2, 3, 4], [5], [6], [8, 9, 10]):
        # two float32 summation orders of the same terms (tests/test_gpu_parity.py's bound for it)
        assert rel_l2(g2[1][:, cols], g2[0][:, cols]) <= 1e-5, cols

