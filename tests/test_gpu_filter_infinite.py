"""An infinite pixel in the feature-guided filter: every window that holds it
averages to that infinity (weights are positive), wherever in the window it
lies, and no other window changes; the same for the adjoint's gradient."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius", [0, 1, 2, 5, 8])
@pytest.mark.parametrize("value", [np.inf, -np.inf])
@pytest.mark.parametrize("shape,at", [((21, 37), (10, 18)), ((21, 37), (0, 0)), ((21, 37), (20, 36)), ((3, 17), (1, 15))])
def test_infinite_pixel_stays_infinite(radius, value, shape, at):
    torch = need_cuda()
    H, W = shape
    rng = np.random.default_rng(radius)
    p = dpcs.make_denoise_params(radius=radius, sigma_s=2.5, sigma_albedo=0.4, sigma_normal=0.6, sigma_depth=0.3)
    d = lambda x: torch.from_numpy(x).cuda()
    guide = d(rng.uniform(0.0, 0.3, (H, W, 8)).astype(np.float32))  # exponents above -60: no weight is 0
    img = rng.uniform(0.5, 2.0, (H, W, 3)).astype(np.float32)
    bad = img.copy()
    bad[at] = value
    c = dpcs.Context(0)
    try:
        out, wsum = c.denoise(d(img), guide, p)
        got, _ = c.denoise(d(bad), guide, p)
        back, back0 = c.denoise_backward(d(bad), guide, wsum, p), c.denoise_backward(d(img), guide, wsum, p)
        c.sync()
        out, got, back, back0 = (x.cpu().numpy() for x in (out, got, back, back0))
    finally:
        c.close()
    y, x = np.mgrid[0:H, 0:W]
    held = (abs(y - at[0]) <= radius) & (abs(x - at[1]) <= radius)
    for new, old in ((got, out), (back, back0)):
        np.testing.assert_array_equal(new[held], value)
        np.testing.assert_array_equal(new[~held], old[~held])
