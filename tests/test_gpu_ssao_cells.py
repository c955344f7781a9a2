"""The pixel that an occlusion sample falls into follows from the rounding of its position, so the paired form of the
positions must round as the scalar sums do: at the pixels below a sample lies within an ulp of a pixel-grid line, and
another order of the fused products moves it across (the second value)."""
import numpy as np
import pytest

from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H = 1024, 768
# view, x, y, occlusion of the scalar sums, of the other order
PINS = [(89, 988, 214, 0.8621054887771606, 0.8998458385467529), (156, 916, 10, 0.8125, 0.75),
        (183, 105, 136, 1.0, 0.9375), (502, 309, 143, 0.9375, 0.875), (530, 429, 76, 0.6875, 0.75),
        (643, 220, 64, 0.31888484954833984, 0.38138484954833984)]


@pytest.fixture(scope="module")
def renderer():
    import torch

    import paper_2501_12750_gb300 as vtx
    rng = np.random.default_rng(9)
    n = 6000
    box = scenes.box_edge(n)
    pos = scenes.protein_like(rng, n, box)
    elem = scenes.draw_elements(rng, n)
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(scenes.pack_xyzr(pos, elem)).cuda(), torch.from_numpy(elem).cuda())
    return r, box


@pytest.mark.parametrize("view,x,y,ao,other", PINS)
def test_samples_on_grid_lines(renderer, view, x, y, ao, other):
    import torch

    import paper_2501_12750_gb300 as vtx
    r, box = renderer
    r.set_camera(scenes.orbit_camera(np.array([box / 2] * 3), box * (0.55 + 0.0005 * view), 7.3 * view,
                                     0.1 * (view % 600) - 30.0, W, H))
    s = vtx.default_settings(ssao_kernel=scenes.ssao_kernel(), flags=vtx.FLAG_SYNC)
    got = float(r.render_frame(s, width=W, height=H)["ao"][y, x])
    torch.cuda.synchronize()
    # 16 samples of weight 1 or less, summed in FP32: 1e-5 is far above the sum's rounding, far below one sample
    assert abs(got - ao) < 1e-5 < abs(other - ao)
