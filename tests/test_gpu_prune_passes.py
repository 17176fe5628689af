"""Pruning's selection, compaction map and compaction at the edges of their
digits, chunks and vector loads, bit for bit against sorting on the host."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2510_06644_gb300 import gs
    gs.lib()
    return gs


def _terms(n, kind, rng):
    t = np.exp(rng.normal(-9.0, 2.0, (n, 2))).astype(np.float32)
    if kind == "ties":      # whole digits of the id decide
        t[:] = np.float32(0.25)
    elif kind == "zeros":   # most were never blended
        t[rng.random(n) < 0.8] = 0.0
    elif kind == "special":
        t[rng.random(n) < 0.3] = np.inf
        t[rng.random(n) < 0.2, 1] = 3e38
    return t


def _select(t, mask, frac, cap):
    s = (t[:, 0] + (np.float32(0.8) * t[:, 1]).astype(np.float32)).astype(np.float32)
    key = (s.view(np.uint32).astype(np.uint64) << np.uint64(32)) | np.arange(len(s), dtype=np.uint64)
    live = np.flatnonzero(mask == 0)
    m = min(int(np.floor(float(np.float32(frac)) * len(live))), cap, len(live))
    out = mask.copy()
    if m > 0:
        out[live[np.argsort(key[live], kind="stable")[:m]]] = 1
    return out


@pytest.mark.parametrize("kind", ["plain", "ties", "zeros", "special"])
@pytest.mark.parametrize("n,frac,cap", [(1, 1.0, 1), (2, 0.5, 2), (2047, 0.1, 2047), (2048, 0.5, 2048),
                                        (2049, 0.999, 2049), (70001, 0.1, 70001), (70001, 0.9, 123),
                                        (70001, 1.0, 70001), (70001, 2.0, 70001), (70001, 0.3, 0)])
@pytest.mark.parametrize("off", [0, 1])
def test_selection(G, n, frac, cap, kind, off):
    rng = np.random.default_rng(n + 17 * off)
    t = _terms(n, kind, rng)
    mask = np.where(rng.random(n) < 0.1, 255, 0).astype(np.uint8)
    td = torch.empty(n * 2 + off, device="cuda")[off:].view(n, 2)  # off: no vector loads
    md = torch.empty(n + off, dtype=torch.uint8, device="cuda")[off:]
    td.copy_(torch.from_numpy(t))
    md.copy_(torch.from_numpy(mask))
    assert G.gs_prune(G.default_config(prune_frac=frac), td, md, 0, 5, max_select=cap) == 5
    assert np.array_equal(md.cpu().numpy(), _select(t, mask, frac, cap))


# 4_300_000 ids make chunks of two steps
@pytest.mark.parametrize("n", [1, 7, 8, 2047, 2048, 2049, 500_003, 4_300_000])
@pytest.mark.parametrize("off", [0, 1])
def test_compaction(G, n, off):
    rng = np.random.default_rng(n)
    mask = np.where(rng.random(n) < 0.3, 7, 0).astype(np.uint8)
    md = torch.empty(n + off, dtype=torch.uint8, device="cuda")[off:]
    md.copy_(torch.from_numpy(mask))
    cmap = torch.empty(n + off, dtype=torch.int32, device="cuda")[off:]
    kept = torch.zeros(1, dtype=torch.int64, device="cuda")
    G.gs_prune(G.default_config(), None, md, 5, 5, change_ratio=0.2, compact_map=cmap, n_kept=kept)
    keep = mask == 0
    exp = np.where(keep, np.cumsum(keep) - 1, -1).astype(np.int32)
    assert int(kept.item()) == keep.sum()
    assert np.array_equal(cmap.cpu().numpy(), exp)
    if n <= 500_003:
        for w in (1, 2, 3, 4, 5):
            src = torch.randn(n, w, device="cuda")
            dst = G.gs_compact(src, cmap, int(keep.sum()))
            assert torch.equal(dst, src[torch.from_numpy(keep).cuda()])
