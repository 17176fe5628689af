"""Opacities that round to 0 (a float16 record's logit below about -17, a
float32 one's below about -88) with alpha_min = 0: such a fragment is blended
with alpha 0, and dL/dopacity = e^(-q/2) T (c . g - s) is an ordinary number.
The masked backward gives the gradients of the kernels without masks, and one
map update leaves the map finite."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import dev, np_of, rel_l2

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


@pytest.mark.parametrize("sx,sy", [(1, 1), (2, 2)])
@pytest.mark.parametrize("rec,logit", [("F16", -20.0), ("F32", -120.0)])
def test_opacity_zero_has_a_finite_gradient(G, rec, logit, sx, sy):
    W, H, n, dt = 368 * sx, 368 * sy, 3000, getattr(G, "GS_" + rec)
    cam = S.camera(W, H, 300.0 * sx, sx=sx, sy=sy)
    g = S.tiny_scene(seed=77, n=n)
    g["log_scales"] += 1.0
    g["opacity_logit"][::3] = logit
    gd, cs, cfg = dev(g), G.camera(cam), G.default_config()
    cfg.alpha_min = 0.0
    rec_t = G.gs_project(cfg, cs, gd, dt)
    cap = int(G.gs_bin_count(cs, rec_t, n, dt, cfg=cfg).item())
    _, vals, _, ranges, order = G.gs_bin_sort(cs, rec_t, n, cap, dt, cfg=cfg)
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    out = G.gs_render_fwd(cfg, cs, rec_t, n, vals, ranges, dt, order=order, masks=bm)
    Ws, Hs, _, _ = G.grid(cam)
    d_rgb, d_dep = (torch.from_numpy(x).cuda() for x in S.image_grads(Ws, Hs, 3))
    g2, grads = [], []
    for k in (None, bm):
        grads.append({q: torch.empty_like(v) for q, v in gd.items()})
        g2.append(np_of(G.gs_render_bwd(cfg, cs, gd, rec_t, vals, ranges, out["t_final"], out["last_idx"], d_rgb,
                                        d_dep, mode=G.GS_MAP, rec_dtype=dt, order=order, masks=k, grads=grads[-1])))
    assert (g2[0][::3, 5] != 0).sum() > 50  # zero opacities that were blended
    assert np.isfinite(g2[0]).all() and np.isfinite(g2[1]).all()
    for cols in ([0, 1], [2, 3, 4], [5], [6], [8, 9, 10]):
        # two float32 summation orders of the same terms (tests/test_gpu_parity.py's bound for it)
        assert rel_l2(g2[1][:, cols], g2[0][:, cols]) <= 1e-5, cols
    assert rel_l2(g2[1][::3, 5], g2[0][::3, 5]) <= 1e-5
    for q, v in grads[1].items():
        assert bool(torch.isfinite(v).all()), q
