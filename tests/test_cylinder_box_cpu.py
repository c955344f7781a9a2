"""CPU emulation (FP32, the kernels' operations) of set-up's candidate pixel box of a bond: no ray that meets the capped
cylinder may have its pixel outside the box.  Eyes far from the origin (the FP32 view centre then carries most of the
error), bonds just beyond the distance where their bounding sphere's box takes over, reciprocals off by their bound."""
import numpy as np
import pytest

F = np.float32
RCP_ERR = 1.2e-7  # relative error of the approximate reciprocal: one ulp


def fma(x, y, z):
    return (np.float64(x) * np.float64(y) + np.float64(z)).astype(F)


def view_f32(basis, d):
    r, u, f = (v.astype(F) for v in basis)
    return [fma(w[0], d[:, 0], fma(w[1], d[:, 1], w[2] * d[:, 2])) for w in (r, u, f)]


@pytest.mark.parametrize("offset", [0.0, 300.0, 20000.0])
@pytest.mark.parametrize("width,height,tan_half", [(1920, 1080, 0.577), (97, 61, 0.2), (3840, 2160, 1.5)])
def test_box_holds_every_hit(offset, width, height, tan_half):
    rng = np.random.default_rng(int(offset) + width)
    n = 60_000
    f = 0.5 * height / tan_half
    cx, cy = 0.5 * width, 0.5 * height
    # an orthonormal basis and an eye, as float32 numbers (the view's constants)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    basis = [c.astype(F) for c in q.T]
    exact = [b.astype(np.float64) for b in basis]
    eye = (offset * rng.standard_normal(3)).astype(F)
    # bonds: 0.1 to 2 A long, near the distance where the box applies and far beyond it
    hl = rng.uniform(0.05, 1.0, n)
    rad = F(rng.choice([0.05, 0.15, 0.5]))
    reach = np.sqrt(hl ** 2 + float(rad) ** 2)
    z = 8.0 * reach * np.where(rng.random(n) < 0.5, 1.0 + 10.0 ** rng.uniform(-5, 0, n), 10.0 ** rng.uniform(0, 2, n))
    slopes = rng.uniform(-1.1, 1.1, (n, 2)) * tan_half * np.array([width / height, 1.0])
    C = np.column_stack([slopes * z[:, None], z]) @ np.stack(exact) + eye
    axis = rng.standard_normal((n, 3))
    axis /= np.linalg.norm(axis, axis=1)[:, None]
    ends = [(C + s * hl[:, None] * axis).astype(F) for s in (-1.0, 1.0)]

    # set-up in FP32
    A, B = ends
    e = B - A
    L = np.sqrt(fma(e[:, 2], e[:, 2], fma(e[:, 0], e[:, 0], e[:, 1] * e[:, 1])))
    inv = F(1.0) / L
    ax, ay, az = ((fma(w[2], e[:, 2], fma(w[0], e[:, 0], w[1] * e[:, 1])) * inv) for w in basis)
    half = F(0.5) * L
    Rb = np.sqrt(fma(half, half, rad * rad)) * F(1.00001)
    c = F(0.5) * (A + B)
    d = c - eye
    vx, vy, vz = view_f32(basis, d)
    err = F(4e-7) * np.abs(d).sum(1, dtype=F) + F(1.2e-7) * np.abs(c).sum(1, dtype=F) + F(1e-6)
    Rm = Rb + err
    used = vz > F(8.0) * Rm
    assert used.mean() > 0.5

    def rcp(x):
        return (1.0 / x.astype(np.float64) * (1.0 + RCP_ERR * rng.choice([-1.0, 1.0], len(x)))).astype(F)

    hc, e0 = F(f * (1.0 + 4e-6)), F(1e-4 + 1e-6 * (width + height))
    rz, rm = rcp(vz), rad + F(2.0) * err + F(1e-5) * Rm
    mx, my = vx * rz, vy * rz
    t = hc * rcp(vz - half * np.abs(az) - rm) * F(1.00001)
    hx = fma(t, fma(half, np.abs(fma(-mx, az, ax)), rm * fma(F(0.5) * mx, mx, F(1.0))), e0)
    hy = fma(t, fma(half, np.abs(fma(-my, az, ay)), rm * fma(F(0.5) * my, my, F(1.0))), e0)
    ux, uy = fma(F(f), mx, F(cx - 0.5)), fma(F(-f), my, F(cy - 0.5))

    # points of the exact capped cylinder of the FP32 ends, 2e-6 wider for the rounding of the hit test itself
    a64, b64 = A.astype(np.float64), B.astype(np.float64)
    mid, half64 = 0.5 * (a64 + b64) - eye.astype(np.float64), 0.5 * np.linalg.norm(b64 - a64, axis=1)
    u64 = (b64 - a64) / (2.0 * half64)[:, None]
    for k in range(24):
        w = np.cross(u64, rng.standard_normal((n, 3)) if k % 3 else np.broadcast_to(exact[k // 3 % 2], (n, 3)))
        w *= (float(rad) * (1.0 + 2e-6) / np.linalg.norm(w, axis=1))[:, None]
        P = mid + (half64 * (1.0 + 2e-6) * rng.choice([-1.0, 1.0, 0.4], n))[:, None] * u64 + w
        p = [P @ v for v in exact]
        px, py = f * p[0] / p[2] + cx - 0.5, -f * p[1] / p[2] + cy - 0.5
        # a pixel whose ray hits is the projection of such a point: none may lie past the box's reach
        assert np.all((np.abs(px - ux) <= hx) & (np.abs(py - uy) <= hy) | ~used)
