"""The bucket sort at the lengths where its paths change (a warp, 128, 256 and
512 threads a bucket, slabs, the merge in global memory), and at depths that
defeat an even distribution: all equal, clustered with outliers, two values,
powers of two.  The result is a function of the keys, so it is exact."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import np_of, pack_splats

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


def depths(kind, n, r):
    if kind == "even":
        d = r.uniform(0.5, 10.0, n)
    elif kind == "equal":
        d = np.full(n, 2.5)
    elif kind == "cluster":  # two thin surfaces and one far Gaussian
        d = np.where(r.random(n) < 0.5, 1.5, 3.0) + 1e-4 * r.normal(size=n)
        d[r.integers(0, n)] = 1e6
    elif kind == "two":
        d = np.where(r.random(n) < 0.5, 1.0, 2.0)
    else:  # spread over many octaves
        d = 2.0 ** r.uniform(-10, 20, n)
    return d.astype(np.float32)


@pytest.mark.parametrize("kind", ["even", "equal", "cluster", "two", "octaves"])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 256, 257, 1024, 1025, 2048, 2049, 4095, 4096, 4097, 8193, 30001, 70001])
def test_bucket_sort_is_exact(G, n, kind):
    W, H = 32, 16  # two tiles: all Gaussians in the left one, a third of them in the right one too
    r = np.random.default_rng(n)
    s = S.splats(n, W, H, seed=3 + n % 97, cull_frac=0.0)
    s["uv"] = np.stack([np.where(np.arange(n) % 3 == 0, 15.5, 6.0), np.full(n, 8.0)], 1).astype(np.float32)
    s["conic"] = np.tile(np.array([[0.8, 0.0, 0.8]], np.float32), (n, 1))
    s["radius"] = np.full(n, 4, np.int32)
    s["opacity"] = np.full(n, 0.9, np.float32)
    s["depth"] = depths(kind, n, r)
    cam = S.camera(W, H, 50.0)
    cap = 2 * n
    keys, vals, nk, ranges, order = G.gs_bin_sort(G.camera(cam), pack_splats(s), n, cap)
    ids = np.arange(n)
    bits = s["depth"].view(np.uint32).astype(np.uint64)
    want_k, want_v = [], []
    for tile, sel in ((0, ids), (1, ids[ids % 3 == 0])):
        o = sel[np.lexsort((sel, bits[sel]))]
        want_k.append((np.uint64(tile) << np.uint64(32)) | bits[o])
        want_v.append(o)
    want_k, want_v = np.concatenate(want_k), np.concatenate(want_v)
    k = int(nk.item())
    assert k == want_k.size
    assert np.array_equal(np_of(keys)[:k].view(np.uint64), want_k)
    assert np.array_equal(np_of(vals)[:k].astype(np.int64), want_v)
