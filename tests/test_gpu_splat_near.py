"""The default splat where its two forms of a hit meet: tiny spheres, which take the short key, and a few that come to the
near or the eye plane with on-screen boxes small enough to be splatted, which do not; with 8, 4 and 1 lanes a survivor."""
import numpy as np
import pytest

from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H, TAN = 61, 48, 1.5
PLANES = ("depth", "id", "normal", "rgb", "ao")


def make(n, near, seed):
    """n spheres of a pixel or two far away, the first `near` of them moved to the eye."""
    rng = np.random.default_rng(seed)
    f = 0.5 * H / TAN
    z = rng.uniform(60.0, 110.0, n)
    p = np.column_stack([rng.uniform(-1, 1, n) * z * TAN * W / H, rng.uniform(-1, 1, n) * z * TAN, z])
    r = rng.uniform(1.2, 1.8, n)
    k = np.arange(near)
    r[k] = rng.uniform(0.05, 0.5, near)
    p[k, 2] = r[k] * rng.uniform(-0.6, 3.0, near) + 0.1
    side = rng.choice([-1.0, 1.0], near)
    p[k, 0] = side * (np.abs(p[k, 2]) * TAN * W / H + r[k] * rng.uniform(0.3, 1.2, near))  # towards the screen's edges
    p[k, 1] = rng.uniform(-1, 1, near) * np.abs(p[k, 2]) * TAN
    order = rng.permutation(n)  # spread over the atoms that the cull samples
    x = np.column_stack([p, r])[order].astype(np.float32)
    size = np.where(x[:, 2] > 8.0 * x[:, 3], x[:, 3] / x[:, 2], 1.0)
    return x, f, size, np.isin(order, k)


@pytest.mark.parametrize("n,near,lanes", [(2000, 10, 8), (24000, 100, 8), (100000, 400, 4), (260000, 1000, 1)])
@pytest.mark.parametrize("mode", ["vdw", "sas"])
def test_near_spheres_among_tiny_ones(n, near, lanes, mode):
    import torch

    import paper_2501_12750_gb300 as vtx
    x, f, size, is_near = make(n, near, n)
    # the library's rule, from all atoms instead of its sample of a quarter: mean box, lanes per survivor
    assert (2.0 * f * np.sqrt(np.mean(size ** 2)) + 1.2) ** 2 < 25.0
    assert lanes == (8 if n <= 49152 else 4 if n <= 163840 else 1)
    eye = np.zeros(3)
    cam = scenes.look_at(eye, np.array([0.0, 0.0, 1.0]), W, H, fovy_deg=float(2.0 * np.degrees(np.arctan(TAN))))
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(x).cuda(), torch.zeros(n, dtype=torch.uint8, device="cuda"))
    r.set_camera(cam)
    kw = dict(mode=vtx.MODE_SAS, probe_radius=0.2, clip_plane=(0.3, 0.0, 1.0, 0.5)) if mode == "sas" else {}
    out = {}
    for splat in (0, 1, 256):
        s = vtx.default_settings(ssao_kernel=scenes.ssao_kernel(), splat_max_px=splat, flags=vtx.FLAG_SYNC, **kw)
        out[splat] = {k: v.cpu().numpy() for k, v in r.render_frame(s, width=W, height=H).items()}
    torch.cuda.synchronize()
    # some of the near spheres that are seen have boxes that are splatted; between the near ones tiny ones are seen
    # (with the probe's radius added, 1,000 near spheres leave no gap)
    ids = out[1]["id"]
    boxes = []
    for i in np.unique(ids[ids >= 0]):
        if is_near[i]:
            y, xx = np.nonzero(ids == i)
            boxes.append((y.max() - y.min() + 1) * (xx.max() - xx.min() + 1))
    assert len(boxes) >= 2 and min(boxes) <= 200
    assert mode == "sas" or (~is_near[ids[ids >= 0]]).any()
    for k in PLANES:
        np.testing.assert_array_equal(out[0][k], out[1][k], err_msg="default, " + k)
        np.testing.assert_array_equal(out[256][k], out[1][k], err_msg="256, " + k)
