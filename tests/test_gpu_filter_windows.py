"""The feature-guided filter at the edges of its windows and tiles."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0, 1, 2, 5, 7, 8])
@pytest.mark.parametrize("shape", [(1, 1), (3, 17), (33, 15), (16, 32)])
def test_filter_windows(orc, radius, shape):
    """The filter's tap pairs at every window edge: odd and even radii, images
    smaller than a window, one column past a tile, and a pixel whose NaN must
    reach the windows that hold it and no other (a window that ends one
    column short of it loads it in a pair).  Tolerances as for the filter's
    other parity tests."""
    torch = need_cuda()
    c = dpcs.Context(0)
    H, W = shape
    rng = np.random.default_rng(100 * radius + W)
    prm = dict(radius=radius, sigma_s=2.5, sigma_albedo=0.4, sigma_normal=0.6, sigma_depth=0.3)
    guide = rng.uniform(0.0, 1.0, (H, W, 8)).astype(np.float32)
    img, dO = rng.uniform(0.0, 2.0, (H, W, 3)).astype(np.float32), rng.normal(size=(H, W, 3)).astype(np.float32)
    p = dpcs.make_denoise_params(**prm)
    d = lambda x: torch.from_numpy(x).cuda()
    try:
        out, wsum = c.denoise(d(img), d(guide), p)
        dI = c.denoise_backward(d(dO), d(guide), wsum, p)
        bad = img.copy()
        by, bx = H // 2, W // 2
        bad[by, bx] = np.nan
        nan, _ = c.denoise(d(bad), d(guide), p)
        c.sync()
        out, wsum, dI, nan = (x.cpu().numpy() for x in (out, wsum, dI, nan))
    finally:
        c.close()
    ref, rden = orc.denoise(img.astype(np.float64), guide.astype(np.float64), prm)
    np.testing.assert_allclose(out, ref, rtol=2e-5, atol=1e-6)
    np.testing.assert_allclose(wsum, rden, rtol=2e-5)
    np.testing.assert_allclose(dI, orc.denoise_backward(dO.astype(np.float64), guide.astype(np.float64), prm), rtol=1e-4, atol=2e-5)
    y, x = np.mgrid[0:H, 0:W]
    held = (abs(y - by) <= radius) & (abs(x - bx) <= radius)
    np.testing.assert_array_equal(np.isnan(nan).any(-1), held)
    np.testing.assert_array_equal(nan[~held], out[~held])
