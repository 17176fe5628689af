"""Gradients of Gaussians smaller than the masked backward's pixel blocks, and
of needles across many of them.  The second-order sums of a small Gaussian (the
conic's gradient) come from few pixels near its own mean, so they keep their
digits only if every pixel's term is formed about that mean; a needle's mean
gradient Q sum h d cancels.  Against the float64 oracle the one-warp masked
kernel may be no farther than twice the kernels without masks, which form the
same terms: both start from the same float32 alphas, whose error (about 2e-7,
at a needle's ends 2e-5) is what separates either from the oracle, and a factor
of two is the room for another order of a few additions."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from synth import scenes as S
from tests.gpu_helpers import dev, np_of, pack_splats, rel_l2

pytestmark = pytest.mark.gpu

SIDE = 376  # sampled pixels a side: 576 to 8836 tiles, so strided frames take the one-warp kernel too


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


def isolated(sigma, aspect, radius, W, H, alpha_min, seed):
    """Gaussians of about `sigma` px and minor / major axes in `aspect`, one in
    every cell of the image, none reaching another's; without those that have
    an alpha within 1e-4 of alpha_min at a pixel, where float32 may decide
    otherwise."""
    g = np.random.default_rng(seed)
    size = 2 * radius + 6
    ny, nx = H // size, W // size
    cell = np.stack(np.meshgrid(np.arange(nx), np.arange(ny)), -1).reshape(-1, 2)
    uv = (size * cell + radius + 1.0 + g.uniform(0, 4, cell.shape)).astype(np.float32)
    n = len(uv)
    s1 = sigma * g.uniform(0.9, 1.1, n)
    s2 = s1 * g.uniform(*aspect, n)
    th = g.uniform(0, np.pi, n)
    c, s = np.cos(th), np.sin(th)
    conic = np.stack([c * c / s1 ** 2 + s * s / s2 ** 2, c * s * (1 / s1 ** 2 - 1 / s2 ** 2),
                      s * s / s1 ** 2 + c * c / s2 ** 2], 1).astype(np.float32)
    op = g.uniform(0.3, 0.9, n).astype(np.float32)
    d = np.arange(-radius, radius + 1)
    px = np.floor(uv.astype(np.float64))[:, None, None, :] + np.stack(np.meshgrid(d, d), -1)[None] + 0.5
    e = px - uv.astype(np.float64)[:, None, None, :]
    A, B, C = (conic[:, k].astype(np.float64)[:, None, None] for k in range(3))
    al = op[:, None, None] * np.exp(-0.5 * (A * e[..., 0] ** 2 + 2 * B * e[..., 0] * e[..., 1] + C * e[..., 1] ** 2))
    ok = ~(np.abs(al / alpha_min - 1.0) < 1e-4).any((1, 2))
    m = int(ok.sum())
    return {"uv": uv[ok], "conic": conic[ok], "opacity": op[ok], "rgb": g.uniform(0.2, 1, (m, 3)).astype(np.float32),
            "depth": g.uniform(0.5, 5, m).astype(np.float32), "radius": np.full(m, radius, np.int32)}


@pytest.mark.parametrize("mode", ["track", "map"])
@pytest.mark.parametrize("sx,sy", [(1, 1), (1, 2), (2, 2), (4, 1), (1, 4), (4, 4)])
@pytest.mark.parametrize("sigma,aspect,radius,near", [
    (0.55, (0.7, 1.0), 4, 1e-5), (0.8, (0.7, 1.0), 4, 1e-5), (1.5, (0.7, 1.0), 4, 1e-5), (12.0, (0.04, 0.06), 36, 5e-5)])
def test_gradients_keep_their_digits(G, sigma, aspect, radius, near, sx, sy, mode):
    cfg = G.default_config()
    W, H = SIDE * sx, SIDE * sy
    cam = S.camera(W, H, 100.0, sx=sx, sy=sy)
    s = isolated(sigma, aspect, radius, W, H, float(cfg.alpha_min), 7)
    rec, n, cs = pack_splats(s), len(s["uv"]), G.camera(cam)
    cap = 100 * n + 64
    _, vals, nk, ranges, order = G.gs_bin_sort(cs, rec, n, cap)
    assert int(nk.item()) <= cap
    bm = torch.zeros(G.gs_blend_mask_words(cs, cap), dtype=torch.int32, device="cuda")
    out = G.gs_render_fwd(cfg, cs, rec, n, vals, ranges, order=order, masks=bm)
    # image gradients of one sign: the terms of a sum do not cancel
    d_rgb, d_dep = (np.abs(x).astype(np.float32) for x in S.image_grads(SIDE, SIDE, 5))
    ref = O.render_bwd(s, cam, d_rgb, d_dep)
    z = dev({"means": np.zeros((n, 3), np.float32), "log_scales": np.zeros((n, 3), np.float32),
             "quats": np.zeros((n, 4), np.float32), "opacity_logit": np.zeros(n, np.float32),
             "rgb": np.zeros((n, 3), np.float32)})
    g2 = [np_of(G.gs_render_bwd(cfg, cs, z, rec, vals, ranges, out["t_final"], out["last_idx"],
                                torch.from_numpy(d_rgb).cuda(), torch.from_numpy(d_dep).cuda(),
                                mode=G.GS_MAP if mode == "map" else G.GS_TRACK, order=order, masks=k))
          for k in (None, bm)]
    assert (ref[:, 2] != 0).sum() > n // 20
    for cols in ([0, 1], [2, 3, 4], [6]) + (([5], [8, 9, 10]) if mode == "map" else ()):
        plain, masked = (rel_l2(g[:, cols], ref[:, cols]) for g in g2)
        assert plain <= near and masked <= 2.0 * plain, (cols, masked, plain)
