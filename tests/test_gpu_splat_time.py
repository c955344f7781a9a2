"""The library-default splat (threshold and lanes per survivor chosen in set-up) against explicit thresholds, on frames
where a wrong choice is dear: many spheres of a few pixels, which gain nothing from shared lanes, and many of ten
pixels across, which the tile raster takes sooner."""
import numpy as np
import pytest

from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu


def fastest(r, out, settings):
    """Microseconds a frame of each of the settings: the least of eleven runs of 40 frames, taken in turn."""
    import torch
    best = [float("inf")] * len(settings)
    for s in settings:
        r.render_frame(s, out=out)
    for _ in range(11):
        for i, s in enumerate(settings):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(40):
                r.render_frame(s, out=out)
            e1.record()
            e1.synchronize()
            best[i] = min(best[i], e0.elapsed_time(e1) * 25.0)
    return best


# explicit threshold that is best there; beside it, the default's time over that threshold's with lanes shared by the
# survivors' number alone and the splat bounded by the number of its pixel tests
@pytest.mark.parametrize("n,w,h,splat", [(48000, 240, 168, 16),    # 1.45
                                         (160000, 340, 237, 16),   # 1.55
                                         (100000, 2560, 1440, 4)])  # 1.2
def test_default_is_near_the_best_threshold(n, w, h, splat):
    import torch

    import paper_2501_12750_gb300 as vtx
    rng = np.random.default_rng(n)
    box = scenes.box_edge(n)
    elem = scenes.draw_elements(rng, n)
    x = scenes.pack_xyzr(scenes.protein_like(rng, n, box), elem)
    c = np.array([box / 2] * 3)
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(x).cuda(), torch.from_numpy(elem).cuda())
    r.set_camera(scenes.look_at(c + np.array([0.0, 0.0, 3.0 * box]), c, w, h))
    out = r.alloc_outputs(w, h)
    r.render_frame(vtx.default_settings(flags=vtx.FLAG_SYNC), out=out)
    explicit, default = fastest(r, out, [vtx.default_settings(splat_max_px=splat), vtx.default_settings()])
    assert default < 1.15 * explicit, (default, explicit)


def test_few_huge_spheres_before_many_small_ones():
    """Out of the middle of a scene of even density: few boxes are huge, most have 4 to 60 pixels. Against an explicit 32;
    with every box splatted, as the mean box of 30 pixels alone suggests, the default took 1.5 times as long."""
    import torch

    import paper_2501_12750_gb300 as vtx
    rng = np.random.default_rng(7)
    n, w, h = 600000, 1280, 720
    z = (20.0 ** 3 + (1500.0 ** 3 - 20.0 ** 3) * rng.random(n)) ** (1.0 / 3.0)
    x = np.empty((n, 4), np.float32)
    x[:, 0] = rng.uniform(-1.03, 1.03, n) * z
    x[:, 1] = rng.uniform(-0.58, 0.58, n) * z
    x[:, 2] = z
    x[:, 3] = 3.0
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(x).cuda(), torch.zeros(n, dtype=torch.uint8, device="cuda"))
    r.set_camera(scenes.look_at(np.zeros(3), np.array([0.0, 0.0, 1.0]), w, h))
    out = r.alloc_outputs(w, h)
    r.render_frame(vtx.default_settings(flags=vtx.FLAG_SYNC), out=out)
    r.render_frame(vtx.default_settings(splat_max_px=32, flags=vtx.FLAG_SYNC), out=out)
    explicit, default = fastest(r, out, [vtx.default_settings(splat_max_px=32), vtx.default_settings()])
    assert default < 1.15 * explicit, (default, explicit)
