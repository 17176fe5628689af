"""Performance cases of the differentiable Gaussian rasterizer: what a SLAM
program has it do, through its public entry points (``gs``, ``pipeline`` and
``autograd``), from the tiny single view to the 3M-Gaussian full-HD frame.

Kinds of case
    track     one tracking iteration (Rasterizer.track_step): projection,
              binning, compositing with the loss, both backwards, pose step.
              A pass is the first iteration of a frame: the pose guess and
              the optimizer state are put in place, then the step runs.
    wave      the same iteration of several sessions in one wave
              (gs_track_wave), mixed map sizes, resolutions and strides.
    map       one mapping iteration to all per-Gaussian gradients
              (Rasterizer.step in GS_MAP mode).
    adam      the map update of a mapping iteration: backward projection with
              the Adam step fused in (gs_project_bwd_adam).
    autograd  gs_render under torch autograd with an L1 loss: forward and
              backward, gradients of the map and of the pose.
    view      rendering a view without gradients (Rasterizer.forward).
    bin       projection, tile intersection and key sort (gs_project_bin_sort).
    interval  the end of a pruning interval: change ratio, selection, removal
              and compaction of the map.

Maps are surface-sampled like an RGB-D SLAM map (planes and spheres, small
log-scales, mostly opaque) or, for the tiny view, uniform in a box.  Targets
are rendered from the true pose; tracking starts 2 cm / 1 degree away.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_06644_gb300 import gs
from paper_2510_06644_gb300.autograd import gs_render
from paper_2510_06644_gb300.pipeline import Rasterizer

PARAMS = ("means", "log_scales", "quats", "opacity_logit", "rgb")
DTYPES = {"f32": gs.GS_F32, "bf16": gs.GS_BF16, "f16": gs.GS_F16}
RESOLUTIONS = ((320, 240), (640, 480), (1200, 680), (1296, 968), (1920, 1080))


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a toy map and image, where launches and latency count
        {"name": "track_tiny_2k_96x72", "kind": "track", "n": 2000, "W": 96, "H": 72, "sx": 1, "sy": 1},
        # the everyday tracking iteration: VGA RGB-D frame, 200k Gaussians
        {"name": "track_200k_640x480", "kind": "track", "n": 200_000, "W": 640, "H": 480, "sx": 1, "sy": 1},
        # the frame after a keyframe is sampled at a 16th of its pixels
        {"name": "track_4x4_97k_640x480", "kind": "track", "n": 97_003, "W": 640, "H": 480, "sx": 4, "sy": 4},
        # later frames of an interval at a quarter of the pixels, larger map and image
        {"name": "track_2x2_458k_1200x680", "kind": "track", "n": 458_001, "W": 1200, "H": 680, "sx": 2, "sy": 2},
        # serving: one iteration of six sessions in one wave
        {"name": "wave_6_sessions", "kind": "wave", "sessions": 6, "n_min": 50_000, "n_max": 600_000},
        # the mapping window's iteration: a keyframe at full resolution, 1M Gaussians
        {"name": "map_1M_1200x680", "kind": "map", "n": 1_000_000, "W": 1200, "H": 680},
        # the map update after it, on a larger map
        {"name": "adam_1500k", "kind": "adam", "n": 1_500_001, "W": 1200, "H": 680},
        # differentiation with 16-bit records on a full-HD frame: the largest work
        {"name": "autograd_f16_3M_1920x1080", "kind": "autograd", "n": 3_000_000, "W": 1920, "H": 1080,
         "rec": "f16", "recompute": False},
        # differentiation of a small odd-sized view with the forward recomputed
        {"name": "autograd_f32_60k_321x239", "kind": "autograd", "n": 60_013, "W": 321, "H": 239, "rec": "f32",
         "recompute": True},
        # inspecting the map: a rendered view, bf16 records
        {"name": "view_bf16_750k_1296x968", "kind": "view", "n": 750_000, "W": 1296, "H": 968, "rec": "bf16"},
        # projection and sorting alone, at the largest tile grid
        {"name": "bin_3M_1920x1080", "kind": "bin", "n": 3_000_000, "W": 1920, "H": 1080, "rec": "f32"},
        # pruning at the end of an interval
        {"name": "interval_1M", "kind": "interval", "n": 1_000_000, "W": 1200, "H": 680},
    ]


def draw(rng):
    def count(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("track", "track", "track", "wave", "map", "adam", "autograd", "view", "bin", "interval"))
    if kind == "wave":
        lo = count(10_000, 100_000)
        return {"kind": kind, "sessions": rng.randint(2, 8), "n_min": lo, "n_max": count(2 * lo, 600_000)}
    W, H = rng.choice(RESOLUTIONS)
    W, H = W + rng.randint(-15, 0), H + rng.randint(-15, 0)
    if kind == "track":
        sx, sy = rng.choice(((1, 1), (1, 1), (2, 2), (4, 2), (4, 4)))
        return {"kind": kind, "n": count(2000, 1_000_000), "W": W, "H": H, "sx": sx, "sy": sy}
    c = {"kind": kind, "n": count(20_000, 2_000_000), "W": W, "H": H}
    if kind in ("autograd", "view", "bin"):
        c["rec"] = rng.choice(("f32", "bf16", "f16"))
    if kind == "autograd":
        c["recompute"] = rng.random() < 0.3
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _camera(W, H, sx=1, sy=1, R=None, t=None):
    f = 80.0 * W / 96.0 if W < 200 else 525.0 * W / 640.0
    return {"R": np.eye(3) if R is None else R, "t": np.zeros(3) if t is None else t, "fx": f, "fy": f,
            "cx": W / 2.0, "cy": H / 2.0, "W": W, "H": H, "sx": sx, "sy": sy}


def _moved(cam, seed, trans=0.02, rot_deg=1.0):
    """The camera moved by `trans` metres and turned by `rot_deg` degrees."""
    r = np.random.default_rng(seed)
    d, ax = r.normal(size=3), r.normal(size=3)
    d, ax = d / np.linalg.norm(d), ax / np.linalg.norm(ax)
    K = np.array([[0, -ax[2], ax[1]], [ax[2], 0, -ax[0]], [-ax[1], ax[0], 0]])
    a = math.radians(rot_deg)
    Rd = np.eye(3) + math.sin(a) * K + (1 - math.cos(a)) * K @ K
    return dict(cam, R=Rd @ cam["R"], t=Rd @ cam["t"] + trans * d)


def _scene(n, seed, box=False):
    """Map of n Gaussians: 70 % on six 4x4 m planes 1-6 m ahead, 30 % on four
    spheres, 1 cm jitter; box: uniform in a box 2-5 m ahead, larger scales."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))

    def uni(*shape, lo=0.0, hi=1.0):
        return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo

    def nrm(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    if box:
        lo, hi = torch.tensor([-1.0, -1.0, 2.0], device="cuda"), torch.tensor([1.0, 1.0, 5.0], device="cuda")
        means, rgb = lo + (hi - lo) * uni(n, 3), uni(n, 3)
        mu, sd, lg = -3.0, 0.3, nrm(n)
    else:
        # planes: centre, two in-plane axes; spheres: centre, radius
        c = torch.stack([uni(6, lo=-1.5, hi=1.5), uni(6, lo=-1.0, hi=1.0), uni(6, lo=1.0, hi=6.0)], 1)
        nv = torch.cat([uni(6, 2, lo=-0.6, hi=0.6), -torch.ones(6, 1, device="cuda")], 1)
        nv = nv / nv.norm(dim=1, keepdim=True)
        up = torch.tensor([0.0, 1.0, 0.0], device="cuda").expand(6, 3)
        a = torch.linalg.cross(nv, up)
        a = a / a.norm(dim=1, keepdim=True)
        b = torch.linalg.cross(nv, a)
        sc = torch.stack([uni(4, lo=-1.2, hi=1.2), uni(4, lo=-0.8, hi=0.8), uni(4, lo=2.0, hi=5.0)], 1)
        rad = uni(4, lo=0.2, hi=0.6)
        base, freq, ph = uni(10, 3, lo=0.15, hi=0.85), uni(6, 3, lo=1.0, hi=4.0), uni(6, 3, lo=0.0, hi=6.0)
        on_plane = uni(n) < 0.7
        ip = torch.randint(0, 6, (n,), generator=g, device="cuda")
        # spheres by area
        cdf = torch.cumsum(rad.square() / rad.square().sum(), 0)
        isp = torch.searchsorted(cdf, uni(n)).clamp(max=3)
        s = uni(n, 2, lo=-2.0, hi=2.0)
        pp = c[ip] + s[:, :1] * a[ip] + s[:, 1:] * b[ip]
        cp = base[ip] + 0.15 * torch.sin(freq[ip] * s[:, :1] + 2.0 * s[:, 1:] + ph[ip])
        d = nrm(n, 3)
        d = d / d.norm(dim=1, keepdim=True)
        ps, cs = sc[isp] + rad[isp, None] * d, base[6 + isp] + 0.15 * d[:, [1, 2, 0]]
        means = torch.where(on_plane[:, None], pp, ps) + 0.01 * nrm(n, 3)
        rgb = (torch.where(on_plane[:, None], cp, cs) + uni(n, 3, lo=-0.1, hi=0.1)).clamp(0, 1)
        mu, sd, lg = -4.5, 0.5, 2.0 + nrm(n)
    q = nrm(n, 4)
    return {"means": means.contiguous(), "log_scales": mu + sd * nrm(n, 3),
            "quats": q / q.norm(dim=1, keepdim=True), "opacity_logit": lg, "rgb": rgb.contiguous()}


def _rasterizer(g, cam, rec=gs.GS_F32):
    """A rasterizer with room for the keys of views near `cam`."""
    n = int(g["means"].shape[0])
    cfg = gs.default_config()
    cs = gs.camera(cam)
    keys = int(gs.gs_bin_count(cs, gs.gs_project(cfg, cs, g, rec), n, rec, cfg=cfg).item())
    return Rasterizer(n, cam, cfg, rec, capacity=int(1.5 * keys) + 4096)


def _observed(r, g, cam):
    """The RGB-D frame of the map from `cam` (0 depth: nothing measured)."""
    img = r.forward(g, cam)
    return img["rgb"].clone(), img["depth"].clone()


def _sessions(case):
    """Sessions of a wave: (n, camera) of each."""
    k = case["sessions"]
    ns = np.exp(np.linspace(math.log(case["n_min"]), math.log(case["n_max"]), k))
    strides, sizes = ((1, 1), (4, 4), (4, 2), (2, 2)), RESOLUTIONS[:3]
    out = []
    for i in range(k):
        W, H = sizes[i % 3]
        sx, sy = strides[i % 4]
        out.append((int(ns[i]), _camera(W, H, sx, sy)))
    return out


def _start(poses):
    """[len(poses), 25] float32: per session the pose guess (12) and a zero
    Adam state (13)."""
    return torch.stack([torch.cat([p, torch.zeros(13, device="cuda")]) for p in poses])


def _tracking(n, cam, seed):
    """Map, camera away from the true pose, observation, rasterizer."""
    g = _scene(n, seed, box=cam["W"] < 200)
    r = _rasterizer(g, cam)
    target = _observed(r, g, cam)
    return g, _moved(cam, seed + 1), target, r


def prepare(case, seed):
    kind = case["kind"]
    if kind == "wave":
        st = {"keep": [], "jobs": [], "guess": []}
        parts = [_tracking(n, cam, seed + 31 * i) for i, (n, cam) in enumerate(_sessions(case))]
        st["guess"] = _start([gs.pose_tensor(cam) for _, cam, _, _ in parts])
        st["state"] = st["guess"].clone()
        for i, (g, cam, target, r) in enumerate(parts):
            pose, adam = st["state"][i, :12], st["state"][i, 12:]
            st["jobs"].append(r.track_job(g, gs.camera(cam, pose=pose), *target, pose, adam))
            st["keep"].append((g, target, r))
        st["cfg"] = gs.default_config()
        return st
    cam = _camera(case["W"], case["H"], case.get("sx", 1), case.get("sy", 1))
    n = case["n"]
    if kind == "track":
        g, cam, target, r = _tracking(n, cam, seed)
        st = {"g": g, "target": target, "r": r, "guess": _start([gs.pose_tensor(cam)])}
        st["state"] = st["guess"].clone()
        st["pose"], st["adam"] = st["state"][0, :12], st["state"][0, 12:]
        st["cam"] = gs.camera(cam, pose=st["pose"])
        return st
    rec = DTYPES[case.get("rec", "f32")]
    g = _scene(n, seed, box=case["W"] < 200)
    cs = gs.camera(cam)
    if kind == "adam":
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        grad2d = torch.randn(n, gs.GRAD2D_STRIDE, generator=gen, device="cuda") * 1e-5
        grad2d *= torch.rand(n, 1, generator=gen, device="cuda") < 0.4  # most Gaussians are not blended
        return {"cam": cs, "cfg": gs.default_config(), "g": g, "grad2d": grad2d,
                "m": {k: torch.zeros_like(v) for k, v in g.items()},
                "v": {k: torch.zeros_like(v) for k, v in g.items()}, "state": torch.zeros(2, device="cuda"),
                "score": torch.empty(n, 2, device="cuda")}
    if kind == "interval":
        cfg = gs.default_config()
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        # Eq. 7 terms: most Gaussians weigh little, a third nothing at all
        score = torch.randn(n, 2, generator=gen, device="cuda").mul(2.0).sub(9.0).exp()
        score *= torch.rand(n, 1, generator=gen, device="cuda") < 0.66
        mask = torch.zeros(n, dtype=torch.uint8, device="cuda")  # a tenth is masked already
        mask[torch.randperm(n, generator=gen, device="cuda")[: n // 10]] = 1
        return {"cfg": cfg, "g": g, "cam": cs, "moved": gs.camera(_moved(cam, seed + 1, 0.005, 0.2)),
                "binned": gs.gs_project(cfg, cs, g), "score": score, "mask": mask}
    if kind == "autograd":
        r = _rasterizer(g, cam)
        target = _observed(r, g, cam)
        p = {k: v.clone().requires_grad_() for k, v in g.items()}
        # the map being optimised has drifted from the one that was observed
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 5)
        with torch.no_grad():
            p["rgb"] += 0.05 * torch.randn(n, 3, generator=gen, device="cuda")
            p["means"] += 0.002 * torch.randn(n, 3, generator=gen, device="cuda")
        return {"p": p, "delta": torch.zeros(6, device="cuda", requires_grad=True), "cam": cam, "target": target,
                "rec": rec, "budget": 0 if case["recompute"] else None}
    r = _rasterizer(g, cam, rec) if kind != "bin" else Rasterizer(n, cam, rec_dtype=rec, capacity=16 * n)
    st = {"g": g, "r": r, "cam": cs}
    if kind == "map":
        away = _moved(cam, seed + 1, 0.02, 0.5)
        st["target"] = _observed(r, g, away)
        st["grads"] = {k: torch.empty_like(v) for k, v in g.items()}
    elif kind == "bin":
        st["ws"] = gs.workspace(gs.gs_project_bin_sort_workspace(r.cfg, cs, g, rec, r.capacity))
        r.keys.zero_()  # entries past the key count are not written
        r.vals.zero_()
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(st):
    if "jobs" in st:
        st["state"].copy_(st["guess"])
        gs.gs_track_wave(st["cfg"], st["jobs"])
        return {"state": st["state"], "score": [r.score for _, _, r in st["keep"]],
                "rgb": [r.img["rgb"] for _, _, r in st["keep"]],
                "depth": [r.img["depth"] for _, _, r in st["keep"]]}
    if "pose" in st:
        r = st["r"]
        st["state"].copy_(st["guess"])
        r.track_step(st["g"], st["cam"], *st["target"], st["pose"], st["adam"])
        return {"pose": st["pose"], "adam": st["adam"], "score": r.score, **r.img}
    if "grad2d" in st:
        gs.gs_project_bwd_adam(st["cfg"], st["cam"], st["g"], st["grad2d"], st["m"], st["v"], st["state"], lr=1e-4,
                               score=st["score"])
        return {"g": st["g"], "m": st["m"], "v": st["v"], "step": st["state"][:1], "score": st["score"]}
    if "binned" in st:
        cfg, g, mask = st["cfg"], st["g"], st["mask"].clone()
        n = mask.numel()
        now = gs.gs_project(cfg, st["moved"], g)
        ratio = gs.gs_change_ratio(st["moved"], st["binned"], now, n, cfg=cfg)
        K = gs.gs_prune(cfg, st["score"], mask, 0, cfg.k0)
        cmap = torch.empty(n, dtype=torch.int32, device="cuda")
        kept = torch.zeros(1, dtype=torch.int64, device="cuda")
        K = gs.gs_prune(cfg, st["score"], mask, K, K, change_ratio=float(ratio.item()), compact_map=cmap, n_kept=kept)
        k = int(kept.item())
        return {"K": K, "ratio": ratio, "mask": mask, "map": cmap, "g": {p: gs.gs_compact(g[p], cmap, k) for p in PARAMS}}
    if "delta" in st:
        p = st["p"]
        rgb, depth = gs_render(*[p[k] for k in PARAMS], st["delta"], st["cam"], rec_dtype=st["rec"],
                               memory_budget=st["budget"])
        loss = (rgb - st["target"][0]).abs().mean() + 0.5 * (depth - st["target"][1]).abs().mean()
        grads = torch.autograd.grad(loss, [*[p[k] for k in PARAMS], st["delta"]])
        return {"rgb": rgb.detach(), "depth": depth.detach(), "grads": dict(zip((*PARAMS, "pose"), grads))}
    r = st["r"]
    if "grads" in st:
        r.step(st["g"], st["cam"], *st["target"], mode=gs.GS_MAP, grads=st["grads"])
        return {"loss": r.dimg["loss"], "grads": st["grads"], "score": r.score, **r.img}
    if "ws" in st:
        gs.gs_project_bin_sort(r.cfg, st["cam"], st["g"], r.splats, r.capacity, r.rec_dtype, ws=st["ws"], keys=r.keys,
                               vals=r.vals, n_keys=r.n_keys, ranges=r.ranges, order=r.order)
        return {"keys": r.keys, "vals": r.vals, "n_keys": r.n_keys, "ranges": r.ranges, "order": r.order,
                "records": r.splats}
    return dict(r.forward(st["g"], st["cam"]))


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: every input read once, every output written once (parameters 56
    bytes a Gaussian, images 16 or 20 bytes a pixel, a record 48 or 32).
    Flops: about 40 blended fragments a pixel (fewer where the map is
    small), 27 in the forward and 67 in the backward, and 200 a Gaussian for
    the projection, 400 for its backward."""
    kind = case["kind"]
    if kind == "wave":
        w = {"bytes": 0, "flops": 0}
        for n, cam in _sessions(case):
            one = work({"kind": "track", "n": n, **{k: cam[k] for k in ("W", "H", "sx", "sy")}})
            w = {k: w[k] + one[k] for k in w}
        return w
    n = case["n"]
    P = -(-case["W"] // case.get("sx", 1)) * -(-case["H"] // case.get("sy", 1))
    rec = 48 if case.get("rec", "f32") == "f32" else 32
    frags = P * 40.0 * min(1.0, 75.0 * n / (40.0 * case["W"] * case["H"]))
    if kind == "adam":
        return {"bytes": n * (56 + 48 + 112 + 168 + 8), "flops": n * (400 + 14 * 12)}
    if kind == "interval":  # score, mask, map; two record sets; the kept parameters
        return {"bytes": n * (8 + 1 + 4 + 56 + 48 + 56 + 0.8 * 56), "flops": n * 260}
    if kind == "bin":  # 12 bytes a key, one key for each tile under about 3 sigma
        keys = (1.0 + 2.0 * 0.0094 * _camera(case["W"], case["H"])["fx"] / 16.0) ** 2
        return {"bytes": n * (56 + rec + 12 * keys), "flops": n * 250}
    if kind == "view":
        return {"bytes": n * 56 + P * 28, "flops": n * 200 + frags * 27}
    out = 8 if kind == "track" else 56 + (8 if kind == "map" else 0)
    return {"bytes": n * (56 + out) + P * (16 + 16), "flops": n * 600 + frags * 94}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------
NEAR, DILATION, ALPHA_MIN, ALPHA_MAX, T_EPS, LAMBDA = 0.2, 0.3, 1.0 / 255.0, 0.99, 1e-4, 0.8


class _Projected64:
    """Projection of a map in float64, differentiable in the map and in a
    left perturbation of the camera pose."""

    def __init__(self, g, cam):
        self.p = {k: v.detach().double().requires_grad_() for k, v in g.items()}
        R = torch.as_tensor(np.asarray(cam["R"], np.float32).astype(np.float64), device="cuda")
        t = torch.as_tensor(np.asarray(cam["t"], np.float32).astype(np.float64), device="cuda")
        self.xi = torch.zeros(6, dtype=torch.float64, device="cuda", requires_grad=True)
        z0 = torch.zeros((), dtype=torch.float64, device="cuda")
        rho, phi = self.xi[:3], self.xi[3:]
        K = torch.stack([torch.stack([z0, -phi[2], phi[1]]), torch.stack([phi[2], z0, -phi[0]]),
                         torch.stack([-phi[1], phi[0], z0])])
        E = torch.eye(3, dtype=torch.float64, device="cuda") + K
        R, t = E @ R, E @ t + rho
        W, H = cam["W"], cam["H"]
        fx, fy, cx, cy = (float(np.float32(cam[k])) for k in ("fx", "fy", "cx", "cy"))
        p = self.p["means"] @ R.T + t
        x, y, z = p.unbind(1)
        self.visible = z >= NEAR
        z = torch.where(self.visible, z, torch.ones_like(z))
        q = self.p["quats"]
        w, a, b, c = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        Rq = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                          2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                          2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).view(-1, 3, 3)
        M = Rq * self.p["log_scales"].exp()[:, None, :]
        self.sigma = M @ M.transpose(1, 2)
        if self.sigma.requires_grad:
            self.sigma.retain_grad()
        S = R @ self.sigma @ R.T
        lx, ly = 1.3 * 0.5 * W / fx, 1.3 * 0.5 * H / fy
        zero = torch.zeros_like(z)
        J = torch.stack([fx / z, zero, -fx * (x / z).clamp(-lx, lx) / z,
                         zero, fy / z, -fy * (y / z).clamp(-ly, ly) / z], 1).view(-1, 2, 3)
        C = J @ S @ J.transpose(1, 2)
        ca, cb, cc = C[:, 0, 0] + DILATION, 0.5 * (C[:, 0, 1] + C[:, 1, 0]), C[:, 1, 1] + DILATION
        det = ca * cc - cb * cb
        self.xy = torch.stack([fx * x / z + cx, fy * y / z + cy], 1)
        self.conic = torch.stack([cc / det, -cb / det, ca / det], 1)
        self.op = torch.sigmoid(self.p["opacity_logit"])
        self.depth = p[:, 2]
        mid = 0.5 * (ca + cc)
        lmax = mid + (mid * mid - det).clamp(min=0.1).sqrt()
        self.radius = torch.where(self.visible, torch.ceil(3 * lmax.sqrt()), torch.zeros_like(lmax)).detach()

    def splats(self):
        return self.xy, self.conic, self.op, self.depth, self.p["rgb"]

    def score(self):
        """Eq. 7 terms: norms of the gradients of the mean and the covariance."""
        G = self.sigma.grad
        G = 0.5 * (G + G.transpose(1, 2))
        return torch.stack([self.p["means"].grad.norm(dim=1), G.flatten(1).norm(dim=1)], 1).float()


def _composite64(P, cam, target=None, w_rgb=1.0, w_depth=0.5):
    """Image, depth and transmittance in float64, tile by tile; with a target
    also the L1 loss and the gradients of the map and the pose (in P)."""
    W, H, sx, sy = cam["W"], cam["H"], cam["sx"], cam["sy"]
    Ws, Hs = -(-W // sx), -(-H // sy)
    leaves = [s.detach().requires_grad_(target is not None) for s in P.splats()]
    order = torch.argsort(leaves[3].detach().float(), stable=True)
    order = order[P.radius[order] > 0]
    lo = (torch.floor(leaves[0].detach()) - P.radius[:, None])[order]
    hi = (torch.floor(leaves[0].detach()) + P.radius[:, None])[order]
    img = torch.zeros(5, Hs, Ws, dtype=torch.float64, device="cuda")
    img[4] = 1.0
    loss = 0.0
    step = max(4, 16 // max(sx, sy)) if max(sx, sy) > 1 else 16
    npix = Ws * Hs
    for j0 in range(0, Hs, step):
        jj = torch.arange(j0, min(Hs, j0 + step), device="cuda", dtype=torch.float64) * sy
        band = (hi[:, 1] >= jj[0]) & (lo[:, 1] <= jj[-1])
        ob, lb, hb = order[band], lo[band], hi[band]
        for i0 in range(0, Ws, step):
            ii = torch.arange(i0, min(Ws, i0 + step), device="cuda", dtype=torch.float64) * sx
            sel = (hb[:, 0] >= ii[0]) & (lb[:, 0] <= ii[-1])
            idx, l, h = ob[sel], lb[sel], hb[sel]
            xy, conic, op, dep, col = (s[idx] for s in leaves)
            px, py = ii.repeat(len(jj))[:, None], jj.repeat_interleave(len(ii))[:, None]
            inside = (px >= l[:, 0]) & (px <= h[:, 0]) & (py >= l[:, 1]) & (py <= h[:, 1])
            dx, dy = px + 0.5 - xy[:, 0], py + 0.5 - xy[:, 1]
            power = -0.5 * (conic[:, 0] * dx * dx + conic[:, 2] * dy * dy) - conic[:, 1] * dx * dy
            alpha = (op * power.exp()).clamp(max=ALPHA_MAX)
            alpha = torch.where(inside & (power <= 0) & (alpha >= ALPHA_MIN), alpha, torch.zeros_like(alpha))
            after = torch.cumprod(1 - alpha.detach(), 1)
            alpha = torch.where(after >= T_EPS, alpha, torch.zeros_like(alpha))  # the pixel has stopped
            keep = torch.cumprod(1 - alpha, 1)
            T = torch.cat([torch.ones_like(px), keep[:, :-1]], 1) if idx.numel() else alpha
            w = alpha * T
            C, D = w @ col, w @ dep
            js, is_ = slice(j0, j0 + len(jj)), slice(i0, i0 + len(ii))
            shape = (len(jj), len(ii))
            img[:3, js, is_] = C.detach().T.reshape(3, *shape)
            img[3, js, is_] = D.detach().reshape(shape)
            if idx.numel():
                img[4, js, is_] = keep[:, -1].detach().reshape(shape)
            if target is not None:
                tc, td = target[0][:, js, is_].double().reshape(3, -1).T, target[1][js, is_].double().reshape(-1)
                part = w_rgb * (C - tc).abs().sum() / (3 * npix)
                part = part + w_depth * ((D - td).abs() * (td != 0)).sum() / npix
                loss += float(part.detach())
                if idx.numel():
                    part.backward()
    if target is not None:
        grads = [s.grad if s.grad is not None else torch.zeros_like(s) for s in leaves]
        torch.autograd.backward(P.splats(), grads)
    return img, loss


def _images64(img):
    img = img.float()
    return {"rgb": img[:3], "depth": img[3], "t_final": img[4], "last_idx": None, "n_blended": None}


def _adam64(p, m, v, g, step, lr, eps):
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    return p - lr * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + eps), m, v


def exact(case, seed):
    kind = case["kind"]
    n = case.get("n", 0)
    if kind == "wave" or (kind in ("track", "map", "autograd", "view") and
                          (n > 250_000 or case["W"] * case["H"] > 350_000)):
        return None  # minutes in 64 bits
    st = prepare(case, seed)
    if kind == "adam":
        P = _Projected64(st["g"], _camera(case["W"], case["H"]))
        d = st["grad2d"].double() * P.visible[:, None]
        torch.autograd.backward(P.splats(), [d[:, 0:2], d[:, 2:5], d[:, 5], d[:, 6], d[:, 8:11]])
        out = {"g": {}, "m": {}, "v": {}, "step": torch.ones(1, device="cuda"), "score": P.score()}
        for k in PARAMS:
            p, m, v = _adam64(P.p[k].detach(), 0.0, 0.0, P.p[k].grad, 1, 1e-4, 1e-15)
            out["g"][k], out["m"][k], out["v"][k] = p.float(), m.float(), v.float()
        return out
    if kind == "interval":
        cfg, mask = st["cfg"], st["mask"].clone()
        s = st["score"][:, 0] + LAMBDA * st["score"][:, 1]
        ids = torch.nonzero(mask == 0)[:, 0]
        ids = ids[torch.argsort(s[ids], stable=True)]
        mask[ids[: math.floor(float(cfg.prune_frac) * ids.numel())]] = 1
        return {"K": None, "ratio": None, "mask": None, "map": None, "g": {k: st["g"][k][mask == 0] for k in PARAMS}}
    if kind == "bin":
        return None  # whole numbers
    cam = _camera(case["W"], case["H"], case.get("sx", 1), case.get("sy", 1))
    if kind == "track":
        cam = _moved(cam, seed + 1)
        P = _Projected64(st["g"], cam)
        img, _ = _composite64(P, cam, st["target"])
        xi, m, v = _adam64(torch.zeros_like(P.xi), 0.0, 0.0, P.xi.grad, 1, 1e-3, 1e-8)
        rho, phi = xi[:3].cpu().numpy(), xi[3:].cpu().numpy()
        th = float(np.linalg.norm(phi))
        K = np.array([[0, -phi[2], phi[1]], [phi[2], 0, -phi[0]], [-phi[1], phi[0], 0]])
        Rd = np.eye(3) + math.sin(th) / th * K + (1 - math.cos(th)) / th ** 2 * K @ K
        V = np.eye(3) + (1 - math.cos(th)) / th ** 2 * K + (th - math.sin(th)) / th ** 3 * K @ K
        R, t = np.asarray(cam["R"], np.float32).astype(np.float64), np.asarray(cam["t"], np.float32).astype(np.float64)
        pose = torch.as_tensor(np.concatenate([(Rd @ R).ravel(), Rd @ t + V @ rho]), device="cuda").float()
        adam = torch.cat([m, v, torch.ones(1, device="cuda", dtype=torch.float64)]).float()
        return {"pose": pose, "adam": adam, "score": P.score(), **_images64(img)}
    if kind == "view":
        with torch.no_grad():
            img, _ = _composite64(_Projected64(st["g"], cam), cam)
        return _images64(img)
    if kind == "map":
        P = _Projected64(st["g"], cam)
        img, loss = _composite64(P, cam, st["target"])
        return {"loss": torch.tensor([loss], dtype=torch.float64), "grads": {k: P.p[k].grad.float() for k in PARAMS},
                "score": P.score(), **_images64(img)}
    P = _Projected64(st["p"], cam)  # autograd: every pixel's depth counts
    t_rgb, t_dep = st["target"]
    img, _ = _composite64(P, cam, (t_rgb, torch.where(t_dep == 0, torch.full_like(t_dep, 1e-30), t_dep)))
    return {"rgb": img[:3].float(), "depth": img[3].float(),
            "grads": {**{k: P.p[k].grad.float() for k in PARAMS}, "pose": P.xi.grad.float()}}
