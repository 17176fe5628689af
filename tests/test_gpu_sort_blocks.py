"""The bucket sort launches as many CTAs as lists of up to the capacity can
fill: grids whose tiles all sit at the edge of a class of list lengths, mixed
ones and nearly empty ones, with the capacity exactly the count."""
import numpy as np
import pytest
import torch

from synth import scenes as S
from tests.gpu_helpers import np_of, pack_splats

pytestmark = pytest.mark.gpu

TX, TY = 9, 7


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs
    gs.gs_status_reset()
    return gs


def lengths(kind):
    t = np.arange(TX * TY)
    if kind == "mixed":
        return np.array([0, 1, 16, 256, 257, 1024, 1025, 2048, 2049, 4097])[t % 10]
    if kind == "one":
        return np.where(t == 40, 1, 0)
    return np.full(TX * TY, int(kind))


@pytest.mark.parametrize("kind", ["1", "256", "257", "1024", "1025", "2048", "2049", "mixed", "one"])
def test_every_list_is_sorted(G, kind):
    length = lengths(kind)
    tile = np.repeat(np.arange(TX * TY), length)
    n = len(tile)
    r = np.random.default_rng(n)
    r.shuffle(tile)
    s = S.splats(n, 16 * TX, 16 * TY, seed=6, cull_frac=0.0)
    s["uv"] = np.stack([16.0 * (tile % TX) + 8.0, 16.0 * (tile // TX) + 8.0], 1).astype(np.float32)
    s["conic"] = np.tile(np.array([[0.8, 0.0, 0.8]], np.float32), (n, 1))
    s["radius"] = np.full(n, 3, np.int32)
    s["opacity"] = np.full(n, 0.9, np.float32)
    keys, vals, nk, ranges, _ = G.gs_bin_sort(G.camera(S.camera(16 * TX, 16 * TY, 50.0)), pack_splats(s), n, n)
    assert int(nk.item()) == n
    bits = s["depth"].view(np.uint32).astype(np.int64)
    o = np.lexsort((np.arange(n), bits, tile))
    assert np.array_equal(np_of(vals)[:n].astype(np.int64), o)
    assert np.array_equal(np_of(keys)[:n], (tile[o].astype(np.int64) << 32) | bits[o])
