"""DIS fusion where residuals are far apart."""
import numpy as np
import pytest

import paper_2106_07136_gb300 as bd
from gpu_helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", [[2.0 ** e for e in range(40, 62, 3)], [1e3, 2.0 ** 51, 2.0 ** 61],
                                    [2.0 ** 46, 2.0 ** 63, np.inf], [2.0 ** 49, 2.0 ** 52],
                                    [np.float32(1.4142135) * 2.0 ** e for e in range(30)]])
def test_a_large_residual_weighs_what_the_division_gives(values):
    """Whole-pixel patches over columns of the right view that take `values` (the left is 0), so
    that a pixel's residuals are up to 2^22 and more apart: the block route that takes reciprocals
    against the one that divides (one weight of each block other than 1), on the pixels that patch
    does not cover, bit for bit."""
    ps, h, w = 8, 128, 256
    kw = dict(patch_size=ps, overlap=0.75, coarsest_scale=0, finest_scale=0,
              fusion=bd._lib.BDIS_FUSION_DIS)
    ny, nx = bd.grid(h, ps, 0.75)[1], bd.grid(w, ps, 0.75)[1]
    rng = np.random.default_rng(len(values))
    d = rng.integers(0, 24, (2, ny, nx)).astype(np.float32)
    L = np.zeros((2, h, w), np.float32)
    R = np.broadcast_to(rng.choice(np.float32(values), w), (2, h, w)).copy()
    one = np.ones_like(d)
    other, touched = one.copy(), np.zeros((h, w), bool)
    for j in range(0, ny, 4):  # a patch every 8 rows and 32 columns: one in each block at least
        for i in range(3, nx, 16):
            other[:, j, i] = 0.5
            touched[2 * j:2 * j + ps, 2 * i:2 * i + ps] = True
    a, b = (host(bd.densify_level((h, w), bd.default_params(**kw), dev(d), dev(v), None, True,
                                  dev(L), packed(R))) for v in (one, other))
    keep = ~touched
    keep[:, :40] = False  # blocks at the image's left edge test every sample anyway
    assert keep.mean() > 0.4 and np.isfinite(a[:, keep]).mean() > 0.9
    np.testing.assert_array_equal(a[:, keep], b[:, keep])


def packed(R):
    """(value, 0) pairs: samples lie on columns, and a difference of infinities is not a number."""
    return dev(np.stack([R, np.zeros_like(R)], -1))
