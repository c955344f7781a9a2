"""The SES distance pass at the edges of its tiles (32 points along x, 32 x 8 rows) and at every window size that
takes the bit-set pass (K = 1..6) or the three separable passes (K >= 7), bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_ses import check_same, gpu_ses

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2), (31, 33, 7), (32, 32, 8), (33, 31, 9), (65, 40, 17)]


@pytest.mark.parametrize("dims", DIMS, ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8])
def test_ses_window_sizes_at_tile_edges(dims, K):
    """Atoms partly outside the grid, whose border cuts the surface; radii from far below to far above the spacing."""
    h = np.float32(0.43)
    probe = float(np.float32((K - 1.3) * h)) if K > 1 else 0.0
    assert int(oracle.lib().orc_ses_k(np.float32(probe), h)) == K
    rng = np.random.default_rng(100 * K + dims[0])
    size = (np.array(dims) - 1) * float(h)
    n = max(2, int(np.prod(size)) // 40)
    x = np.empty((n, 4), np.float32)
    x[:, :3] = rng.uniform(-1.5, size + 1.5, (n, 3))
    x[:, 3] = rng.uniform(0.05, 2.2, n)
    origin = np.array([0.0, 0.013, -0.007], np.float32)
    d = np.array(dims, np.int32)
    check_same(gpu_ses(x, origin, h, d, probe), oracle.ses(x, origin, h, d, probe=probe), "K=%d %s" % (K, dims))
