"""Soft passes off their common path: images whose width is no multiple of four (empty tiles are filled pixel by pixel),
and more than 131,072 tiles (one unordered tile list instead of one per length class)."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu

TOL = 5e-5  # forward planes against float64 (depth: times the camera's distance), as in the soft parity tests


def scene(n, w, h, views, distance):
    rng = np.random.default_rng(n + w)
    box = scenes.box_edge(n)
    x = scenes.pack_xyzr(scenes.protein_like(rng, n, box), scenes.draw_elements(rng, n))
    c = np.array([box / 2] * 3)
    return x, [scenes.orbit_camera(c, distance * box, 23.0 * k, 7.0 * k - 40.0, w, h) for k in range(views)]


def forward_into_nan(r, x, cams):
    """The forward pass into planes and a state that hold NaN before."""
    import torch

    import paper_2501_12750_gb300 as vtx
    v, h, w = len(cams), cams[0].height, cams[0].width
    cov, dep, nrm, state = (torch.full(s, float("nan"), device="cuda")
                            for s in ((v, h, w), (v, h, w), (v, 3, h, w), (v, h, w, 2)))
    assert r.lib.vtx_render_soft_fwd_ex(r.ctx, ctypes.c_void_p(x.data_ptr()), x.shape[0], vtx.camera_array(cams), v,
                                        ctypes.c_float(0.5), vtx.FLAG_SYNC, *(ctypes.c_void_p(t.data_ptr())
                                                                              for t in (cov, dep, nrm, state))) == 0
    torch.cuda.synchronize()
    return cov, dep, nrm, state


def check_filled(cov, dep, nrm, state):
    import torch
    empty = cov == 0.0
    for p in (cov, dep, nrm):
        assert bool(torch.isfinite(p).all())
    assert float(dep[empty].abs().max()) == 0.0
    assert float(nrm.movedim(1, -1)[empty].abs().max()) == 0.0
    bits = state.view(torch.int32)
    untouched = bits[..., 1] == 0
    assert bool((cov[untouched] == 0.0).all()) and bool((state[..., 0][untouched] == 1.0).all())
    assert float(untouched.float().mean()) > 0.3


@pytest.mark.parametrize("w,h", [(97, 61), (50, 130), (1, 40), (33, 17), (18, 16), (64, 48)])
def test_empty_tiles_of_any_width(w, h):
    import torch

    import paper_2501_12750_gb300 as vtx
    x, cams = scene(300, w, h, 3, 4.0)
    planes = forward_into_nan(vtx.Renderer(), torch.from_numpy(x).cuda(), cams)
    cov, dep, nrm, state = planes
    check_filled(*planes)
    for v, cam in enumerate(cams):
        o = oracle.soft_forward(x.astype(np.float64), cam, oracle.all_pixels(w, h))
        ok = o.flags == 0
        dist = float(np.linalg.norm(np.asarray(cam.eye, np.float64) - x[:, :3].mean(0)))
        assert np.abs(cov[v].cpu().numpy().ravel()[ok] - o.A[ok]).max() <= TOL
        assert np.abs(dep[v].cpu().numpy().ravel()[ok] - o.D[ok]).max() <= TOL * dist
        assert np.abs(nrm[v].cpu().numpy().reshape(3, -1).T[ok] - o.N[ok]).max() <= TOL


@pytest.mark.parametrize("w,h,views", [(1457, 1459, 16), (1460, 1459, 16), (1024, 1024, 4)])
def test_many_tiles(w, h, views):
    """More than 131,072 tiles (a single list), and more lists than the sorting CTAs take at once: the planes, the state
    and the gradients of as many calls of one view each."""
    import torch

    import paper_2501_12750_gb300 as vtx
    x, cams = scene(2500, w, h, views, 1.7)
    assert (views == 4) == (views * (-(-w // 16)) * (-(-h // 16)) <= 131072)
    x = torch.from_numpy(x).cuda()
    r = vtx.Renderer()
    planes = forward_into_nan(r, x, cams)
    check_filled(*planes)
    gen = torch.Generator(device="cuda").manual_seed(5)
    up = [torch.randn(p.shape, generator=gen, device="cuda") for p in planes[:3]]
    grad = {k: r.render_soft_bwd(x, cams, *up, **kw) for k, kw in
            (("lists", dict(state=planes[3], reuse_lists=True)), ("rebuilt", dict(state=planes[3])), ("walk", {}))}
    sums = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    one = vtx.Renderer()
    for v in range(views):
        part = forward_into_nan(one, x, cams[v:v + 1])
        for a, b in zip(planes, part):
            assert torch.equal(a[v].view(torch.int32), b[0].view(torch.int32))
        sums += one.render_soft_bwd(x, cams[v:v + 1], *(u[v:v + 1] for u in up), state=part[3]).double()
    scale = float(sums.norm())
    assert scale > 0.0
    for k, g in grad.items():
        # the same FP32 terms added in another order by atomics: a few thousand additions of unit roundoff 6e-8 each
        assert float((g.double() - sums).norm()) <= 1e-5 * scale, k
