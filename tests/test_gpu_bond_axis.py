"""Bonds decoded by the resolve: their axis has the bits of one written-out formula (a visible cap's normal is the axis),
and every pixel that a bond wins shows a point of the capped cylinder, near grazing rays and rims included.  A ray that
set-up accepts and the resolve misses would show the middle of the bond and the normal of a cap."""
import numpy as np
import pytest

from paper_2501_12750_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H = 1201, 903
BOND_RADIUS = np.float32(0.3)


def fma(x, y, z):
    """FP32 multiply-add through the wider long double (64 or 113 bits: one rounding in practice)."""
    wide = np.longdouble
    return (x.astype(wide) * y.astype(wide) + z.astype(wide)).astype(np.float32)


def dot(a, b):
    """Three products, the second rounded by itself."""
    return fma(a[2], b[2], fma(a[0], b[0], a[1] * b[1]))


@pytest.mark.parametrize("direction", [(0.0, 0.0, 1.0), (0.6, 0.2, 0.77), (-0.5, 0.7, 0.3)])
@pytest.mark.parametrize("splat", [0, 256])  # every bond through the raster, small ones splatted
def test_bond_pixels(direction, splat):
    import torch

    import paper_2501_12750_gb300 as vtx
    rng = np.random.default_rng(3)
    n = 4000
    x = np.empty((n, 4), np.float32)
    x[:, :3] = 60.0 * rng.random((n, 3))
    d = rng.standard_normal((n // 2, 3))
    x[1::2, :3] = x[::2, :3] + (d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(0.8, 1.9, (n // 2, 1))).astype(np.float32)
    x[:, 3] = 1.5
    pairs = np.arange(n, dtype=np.int32).reshape(-1, 2)
    cam = scenes.look_at(np.array([30.3, 30.1, 30.0]) + 40.0 * np.array(direction), np.array([30.0] * 3), W, H)
    r = vtx.Renderer()
    r.upload_atoms(torch.from_numpy(x).cuda(), torch.zeros(n, dtype=torch.uint8, device="cuda"))
    r.upload_bonds(torch.from_numpy(pairs).cuda())
    r.set_camera(cam)
    s = vtx.default_settings(mode=vtx.MODE_BALL_AND_STICK, flags=vtx.FLAG_SYNC, splat_max_px=splat)
    s.ball_radius, s.bond_radius = 0.01, BOND_RADIUS  # the caps stay visible
    out = {k: v.cpu().numpy() for k, v in r.render_frame(s, width=W, height=H).items()}
    torch.cuda.synchronize()
    py, px = np.nonzero(out["id"] >= n)
    assert len(px) > 300_000
    A, B = (x[pairs[out["id"][py, px] - n, k]] for k in (0, 1))
    normal = out["normal"][:, py, px]

    # the axis in FP32
    e = [B[:, k] - A[:, k] for k in range(3)]
    inv = np.float32(1.0) / np.sqrt(dot(e, e))
    axis = [dot([np.full(len(px), w, np.float32) for w in np.asarray(v, np.float32)], e) * inv
            for v in (cam.right, cam.up, cam.forward)]
    axis = np.stack([axis[0], axis[1], -axis[2]])
    cap = np.abs(np.abs((axis * normal).sum(0)) - 1.0) < 1e-6  # no side normal: those are at right angles to the axis
    assert cap.sum() > 50_000
    np.testing.assert_array_equal(np.abs(normal[:, cap]), np.abs(axis[:, cap]))

    # the point in float64: on the side or on a cap
    F, R, U = (np.asarray(v, np.float64) for v in (cam.forward, cam.right, cam.up))
    t = np.float64(cam.tan_half_fovy)
    a = (2.0 * (px + 0.5) - W) / H * t
    b = (H - 2.0 * (py + 0.5)) / H * t
    P = np.asarray(cam.eye, np.float64) + out["depth"][py, px, None].astype(np.float64) * (
        F + a[:, None] * R + b[:, None] * U)
    a3, b3 = A[:, :3].astype(np.float64), B[:, :3].astype(np.float64)
    L = np.linalg.norm(b3 - a3, axis=1)
    u = (b3 - a3) / L[:, None]
    q = P - 0.5 * (a3 + b3)
    axial = (q * u).sum(1)
    radial = np.linalg.norm(q - axial[:, None] * u, axis=1)
    tol = 1e-3  # FP32 depths of 20 to 100 A carry 1e-5, grazing rays and rims up to some 1e-4 along the ray
    side = (np.abs(radial - BOND_RADIUS) < tol) & (np.abs(axial) < 0.5 * L + tol)
    end = (np.abs(np.abs(axial) - 0.5 * L) < tol) & (radial < BOND_RADIUS + tol)
    assert np.all(side | end), "%d of %d" % ((~(side | end)).sum(), len(px))
