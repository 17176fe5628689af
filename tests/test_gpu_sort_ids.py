"""Buckets whose keys all have one depth, sorted through bins of their ids:
ids next to one another, spread over a large map, and crowded beside one far
id (too many a bin: the merge sort)."""
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


@pytest.mark.parametrize("ids", ["dense", "spread", "far"])
@pytest.mark.parametrize("n", [2, 200, 257, 1000, 2049, 4096, 4097, 9000])
def test_one_depth(G, n, ids):
    N = 40 * n + 3
    sel = {"dense": 7 + np.arange(n), "spread": np.sort(np.random.default_rng(n).choice(N, n, replace=False)),
           "far": np.append(np.arange(n - 1), N - 1)}[ids]
    s = S.splats(N, 16, 16, seed=5, cull_frac=0.0)
    s["uv"][:] = 8.0
    s["conic"][:] = np.array([0.8, 0.0, 0.8], np.float32)
    s["opacity"][:] = 0.9
    s["depth"][:] = 2.5
    s["radius"][:] = 0
    s["radius"][sel] = 4
    keys, vals, nk, _, _ = G.gs_bin_sort(G.camera(S.camera(16, 16, 50.0)), pack_splats(s), N, n)
    assert int(nk.item()) == n
    assert np.array_equal(np_of(vals)[:n].astype(np.int64), sel)
    assert np.all(np_of(keys)[:n] == np.float32(2.5).view(np.uint32).astype(np.int64))
