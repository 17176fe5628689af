"""Threads that take many Gaussians: the backward projection in one wave (pose
sums over any number a thread), the fused Adam step, and the counting rows of
large maps."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

PARAMS = ("means", "log_scales", "quats", "opacity_logit", "rgb")


@pytest.fixture(scope="module")
def G():
    from paper_2510_06644_gb300 import gs
    gs.lib()
    return gs


def _scene(n, seed=0):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.rand(*s, generator=gen, device="cuda")  # noqa: E731
    return {"means": torch.cat([r(n, 2) * 4 - 2, r(n, 1) * 4 + 0.5], 1).contiguous(), "log_scales": r(n, 3) - 4.5,
            "quats": r(n, 4) + 0.1, "opacity_logit": r(n) * 4 - 2, "rgb": r(n, 3)}


def _cam(G):
    return G.camera({"R": np.eye(3), "t": np.zeros(3), "fx": 260.0, "fy": 250.0, "cx": 160.0, "cy": 120.0, "W": 320,
                     "H": 240})


def _part(g, a, b):
    return {k: v[a:b].contiguous() for k, v in g.items()}


def _bwd(G, cam, g, grad2d):
    n = g["means"].shape[0]
    out = {k: torch.full_like(v, float("nan")) for k, v in g.items()}
    pose = torch.full((6,), float("nan"), dtype=torch.float64, device="cuda")
    score = torch.full((n, 2), float("nan"), device="cuda")
    G.gs_project_bwd(G.default_config(), cam, g, grad2d, grads=out, pose=pose, score=score)
    return out, pose, score


# 152 SMs x 3 CTAs x 256 threads = 116736: one, two, three and nine a thread
@pytest.mark.parametrize("n", [1, 511, 116737, 233473, 1_000_003])
def test_pose_and_gradients_do_not_depend_on_the_split(G, n):
    g, cam = _scene(n, n), _cam(G)
    gen = torch.Generator(device="cuda").manual_seed(n + 1)
    grad2d = torch.randn(n, G.GRAD2D_STRIDE, generator=gen, device="cuda")
    out, pose, score = _bwd(G, cam, g, grad2d)
    total, size = torch.zeros_like(pose), torch.zeros_like(pose)
    for a in range(0, n, 100_000):
        b = min(n, a + 100_000)
        o, p, s = _bwd(G, cam, _part(g, a, b), grad2d[a:b].contiguous())
        for k in PARAMS:
            assert torch.equal(out[k][a:b], o[k])
        assert torch.equal(score[a:b], s)
        total += p
        size += p.abs()
    # float32 pairs: 2^-45 of the terms' magnitudes and below; the terms' sizes
    # are at least the slices' (n / 1000 leaves room for what cancels in them)
    assert ((pose - total).abs() <= 2.0 ** -45 * (1 + n / 1000) * size.max()).all(), (pose, total)


@pytest.mark.parametrize("n", [1, 255, 257, 40_001])
def test_adam_step_against_float64(G, n):
    """Gradients, moments and values of either sign, zeros (whose step is left
    out) and infinities: the fused step is the update of its own gradients."""
    g, cam = _scene(n, n), _cam(G)
    gen = torch.Generator(device="cuda").manual_seed(n + 1)
    grad2d = torch.randn(n, G.GRAD2D_STRIDE, generator=gen, device="cuda")
    grad2d *= torch.rand(n, 1, generator=gen, device="cuda") < 0.5
    if n > 300:
        grad2d[7] = float("inf")
    m = {k: 0.01 * torch.randn(v.shape, generator=gen, device="cuda") for k, v in g.items()}
    v = {k: 0.01 * torch.rand(x.shape, generator=gen, device="cuda") for k, x in g.items()}
    half = torch.rand(n, generator=gen, device="cuda") < 0.5
    for k in PARAMS:
        m[k][half] = 0.0
        v[k][half] = 0.0
    old = {k: (g[k].double(), m[k].double(), v[k].double()) for k in PARAMS}
    grads = {k: torch.full_like(x, float("nan")) for k, x in g.items()}
    b1, b2, eps, lr, t = 0.9, 0.999, 1e-15, 1e-2, 4.0
    state = torch.tensor([t - 1, 0.0], device="cuda")
    G.gs_project_bwd_adam(G.default_config(), cam, g, grad2d, m, v, state, lr=lr, grads=grads)
    assert state.tolist() == [t, 0.0]
    f = lambda x: float(np.float32(x))  # noqa: E731
    for k in PARAMS:
        d, (p0, m0, v0) = grads[k].double(), old[k]
        mm = f(b1) * m0 + (1 - f(b1)) * d
        vv = f(b2) * v0 + (1 - f(b2)) * d * d
        step = f(lr) / (1 - f(b1) ** t) * mm / ((vv / (1 - f(b2) ** t)).sqrt() + f(eps))
        step = torch.where(mm == 0, torch.zeros_like(step), step)
        fin = torch.isfinite(grads[k]) & torch.isfinite(vv.float())
        # the bias corrections cancel in float32 (1 - 0.999^4 keeps 2^-24 / 4e-3 = 1.5e-5)
        err = (g[k].double() - (p0 - step)).abs()
        assert (err <= 2.0 ** -23 * p0.abs() + 4e-5 * step.abs() + 1e-12)[fin].all(), (k, err[fin].max())
        scale_m = f(b1) * m0.abs() + mm.abs() + 0.1 * grads[k].double().abs()
        assert ((m[k].double() - mm).abs() <= 2.0 ** -21 * scale_m + 1e-37)[fin].all()
        assert ((v[k].double() - vv).abs() <= 2.0 ** -21 * vv + 1e-37)[fin].all()


@pytest.mark.parametrize("n", [466_944, 466_945, 1_200_001])
def test_rows_of_large_maps(G, n):
    """912 rows of 512 Gaussians, then longer rows: the sorted keys are every
    (tile, depth, id) of the records' rects once."""
    g, cam = _scene(n, 3), _cam(G)
    g["log_scales"] -= 1.0
    cfg = G.default_config()
    splats = torch.empty(n, 12, device="cuda")
    cap = 8 * n
    keys, vals, n_keys, ranges, order = G.gs_project_bin_sort(cfg, cam, g, splats, cap)
    k = int(n_keys.item())
    touched = splats[:, 11].view(torch.int32).long()
    assert k == int(touched.sum()) <= cap
    kk, vv = keys[:k], vals[:k].long()
    assert torch.equal(torch.bincount(vv, minlength=n), touched)
    assert torch.equal(kk & 0xFFFFFFFF, splats[:, 6].view(torch.int32).long()[vv])
    later = kk[1:] > kk[:-1]
    assert (later | ((kk[1:] == kk[:-1]) & (vv[1:] > vv[:-1]))).all()
    assert torch.equal(torch.bincount(kk >> 32, minlength=len(ranges)), (ranges[:, 1] - ranges[:, 0]).long())
