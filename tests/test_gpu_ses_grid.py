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


@pytest.mark.parametrize("shift", [0.0, 3000.0, 60000.0])
def test_ses_interior_far_from_the_origin(shift):
    """The FP32 filter of the interior widens with the coordinates until the exact test decides every chord's ends;
    radii that put points exactly on a sphere (grid-aligned centres, R a multiple of the spacing) are decided alike."""
    rng = np.random.default_rng(5)
    x = np.empty((60, 4), np.float32)
    x[:, :3] = np.round(rng.uniform(0, 12, (60, 3)) * 2) / 2 + shift
    x[:30, :3] += rng.uniform(-0.3, 0.3, (30, 3)).astype(np.float32)
    x[:, 3] = rng.choice([0.5, 1.0, 1.5, 1.7], 60)
    origin, d = np.full(3, shift - 4.0, np.float32), np.array((41, 41, 41), np.int32)
    ref = oracle.ses(x, origin, np.float32(0.5), d, probe=1.5)
    g = gpu_ses(x, origin, 0.5, d, 1.5)
    np.testing.assert_array_equal(g["sas"], ref.sas)
    np.testing.assert_array_equal(g["edt2"], ref.edt2)
    np.testing.assert_array_equal(g["labels"], ref.edges)


def test_ses_count_then_emit():
    """The two-call form: no surface before the first count or after a plain call; partial and repeated writes; the
    distances also go to the caller's plane."""
    import ctypes

    import torch

    import paper_2501_12750_gb300 as vtx
    rng = np.random.default_rng(3)
    x = torch.from_numpy(np.concatenate([rng.uniform(0, 8, (30, 3)), rng.uniform(1, 2, (30, 1))], 1)
                         .astype(np.float32)).cuda()
    r = vtx.Renderer()
    g = r.ses_fit_grid(x, probe=1.4, spacing=0.5)
    ref = r.ses_mesh(x, g, max_tris=20000, labels=True, planes=True)
    n = ctypes.c_int64(0)
    buf = torch.zeros((ref["n"], 3, 3), device="cuda")
    assert r.lib.vtx_ses_emit(r.ctx, buf.data_ptr(), ref["n"], None) == 7  # VTX_ERR_STATE
    edt = torch.empty_like(ref["edt2"])
    assert r.lib.vtx_ses_count(r.ctx, x.data_ptr(), 30, ctypes.byref(g), None, edt.data_ptr(), ctypes.byref(n)) == 0
    assert n.value == ref["n"] and torch.equal(edt, ref["edt2"])
    edt.zero_()  # the caller's plane is its own again
    part = torch.zeros((100, 3, 3), device="cuda")
    assert r.lib.vtx_ses_emit(r.ctx, part.data_ptr(), 100, None) == 4  # VTX_ERR_CAPACITY
    assert torch.equal(part, ref["tris"][:100])
    assert r.lib.vtx_ses_emit(r.ctx, buf.data_ptr(), n.value, None) == 0
    assert torch.equal(buf, ref["tris"])
    full = r.ses_mesh(x, g, labels=True)
    assert torch.equal(full["tris"], ref["tris"]) and torch.equal(full["labels"], ref["labels"])
