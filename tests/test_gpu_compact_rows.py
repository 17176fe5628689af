"""Compaction of arrays of one to five floats a row at the edges of the rows a
block moves, and over more blocks than the launch has."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 511, 513, 1023, 1024, 1025, 70_001, 12_000_003])
def test_compact_keeps_the_unmasked_rows(n, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs as G
    n = min(n, 36_000_000 // width)
    gen = torch.Generator(device="cuda").manual_seed(n)
    src = torch.rand(n, width, generator=gen, device="cuda")
    keep = torch.rand(n, generator=gen, device="cuda") < 0.7
    k = int(keep.sum())
    cmap = torch.where(keep, torch.cumsum(keep, 0) - 1, torch.full((n,), -1, device="cuda")).to(torch.int32)
    assert torch.equal(G.gs_compact(src, cmap, k), src[keep])
