"""The library-default direct splat (threshold and lanes per survivor chosen in set-up) gives the planes of the fully
binned frame, bit for bit, in every regime: 8, 4 and 1 lanes per survivor, a few primitives, spheres that reach the
eye plane (whose keys are clamped), SAS radii with a clip plane; and the odd sizes of the RGBA8 export."""
import numpy as np
import pytest

from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu

PLANES = ("depth", "id", "normal", "rgb", "ao")


def planes(x, elem, cam, **kw):
    import torch

    import paper_2501_12750_gb300 as vtx
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(x).cuda(), torch.from_numpy(elem).cuda())
    r.set_camera(cam)
    s = vtx.default_settings(ssao_kernel=scenes.ssao_kernel(), flags=vtx.FLAG_SYNC, **kw)
    out = r.render_frame(s, width=cam.width, height=cam.height)
    torch.cuda.synchronize()
    return {k: out[k].cpu().numpy() for k in PLANES}


# atoms, image, distance in box edges: 8 lanes (one warp, ragged warps), 4 lanes, 1 lane, and a crowded image
CASES = [(1, 40, 31, 3.0), (33, 97, 61, 2.0), (2001, 333, 207, 2.0), (20011, 640, 479, 3.0), (70001, 801, 600, 3.0),
         (200003, 641, 480, 3.0), (900, 160, 120, 0.6), (3000, 255, 131, 0.3)]


@pytest.mark.parametrize("n,w,h,dist", CASES)
def test_default_splat_equals_binned(n, w, h, dist):
    rng = np.random.default_rng(n)
    box = scenes.box_edge(max(n, 100))
    pos = scenes.protein_like(rng, n, box)
    elem = scenes.draw_elements(rng, n)
    x = scenes.pack_xyzr(pos, elem)
    c = np.array([box / 2] * 3)
    cam = scenes.look_at(c + np.array([0.1, 0.2, dist * box]), c, w, h)
    import paper_2501_12750_gb300 as vtx
    for kw in ({}, dict(mode=vtx.MODE_SAS, clip_plane=(0.0, 0.3, -1.0, 0.7 * box))):
        ref = planes(x, elem, cam, splat_max_px=1, **kw)
        got = planes(x, elem, cam, **kw)
        assert n < 100 or (ref["id"] >= 0).any()
        for k in PLANES:
            np.testing.assert_array_equal(got[k], ref[k], err_msg="%s %s" % (k, kw))


@pytest.mark.parametrize("w,h,n,skew", [(4, 4, 1, 0), (7, 5, 3, 0), (64, 33, 2, 1), (62, 31, 2, 0), (256, 9, 1, 3)])
def test_export_sizes_and_alignments(w, h, n, skew):
    """One and four pixels per thread: odd pixel counts, image batches, an image that is not 16-byte aligned."""
    import torch

    import paper_2501_12750_gb300 as vtx
    gen = torch.Generator(device="cuda").manual_seed(w * h)
    rgb = torch.rand((n, 3, h, w), generator=gen, device="cuda") * 1.4 - 0.2
    ids = torch.randint(-1, 3, (n, h, w), generator=gen, device="cuda", dtype=torch.int32)
    rgba = torch.zeros(4 * n * h * w + 16, dtype=torch.uint8, device="cuda")[4 * skew:4 * skew + 4 * n * h * w]
    vtx.Renderer().export_rgba8({"rgb": rgb, "id": ids}, background_alpha=0.3, rgba=rgba)
    want = torch.empty((n, h, w, 4), dtype=torch.uint8, device="cuda")
    want[..., :3] = (rgb.clamp(0.0, 1.0) * 255.0).round().permute(0, 2, 3, 1).to(torch.uint8)
    want[..., 3] = torch.where(ids >= 0, 255, 76).to(torch.uint8)
    assert torch.equal(rgba.reshape(n, h, w, 4), want)
