"""gs_adam where an element's first moment is 0 or something is not finite: an
element without momentum keeps its value bit for bit, and infinities and NaN
come out as the formula gives them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_zero_momentum_and_non_finite_elements():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_06644_gb300 import build
    build.build()
    from paper_2510_06644_gb300 import gs as G
    inf, nan, f = np.inf, np.nan, np.float32
    p = np.array([1.5, -0.0, 2.0, 3.0, 4.0, 5.0, 6.0, 7.0, inf, nan, 8.0], f)
    g = np.array([0.0, 0.0, 0.0, 0.0, 0.0, inf, -inf, nan, 0.0, 0.0, 1e-3], f)
    m = np.array([0.0, 0.0, 0.0, 0.0, nan, 0.0, 0.0, 0.0, 0.0, 0.0, 0.1], f)
    v = np.array([0.0, 0.0, 0.5, nan, 0.1, 0.1, 0.1, 0.1, 0.0, 0.0, 0.1], f)
    lr, b1, b2, eps = (f(x) for x in (1e-3, 0.9, 0.999, 1e-8))
    with np.errstate(all="ignore"):
        m1 = (b1 * m + (f(1) - b1) * g).astype(np.float64)
        v1 = (b2 * v + (f(1) - b2) * g * g).astype(np.float64)
        want = p - float(lr) * (m1 / (1 - float(b1))) / (np.sqrt(v1 / (1 - float(b2))) + float(eps))
    t = [torch.from_numpy(x.copy()).cuda() for x in (p, g, m, v)]
    G.gs_adam([t[0]], [t[1]], [t[2]], [t[3]], torch.zeros(2, device="cuda"), lr=1e-3)
    got = t[0].cpu().numpy()
    still = (m == 0) & (g == 0) & ~np.isnan(v)
    assert np.array_equal(got[still].view(np.uint32), p[still].view(np.uint32))
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.isnan(want).sum() == 6
    ok = np.isfinite(want)
    assert np.allclose(got[ok], want[ok], rtol=1e-6, atol=0)
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
