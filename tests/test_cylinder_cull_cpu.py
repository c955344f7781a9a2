"""CPU emulation (FP32, the kernels' operations) of what lets the renderer skip a bond cylinder: the per-axis pixel
reach of its candidate boxes, and the hit test's early return.  Neither may drop a ray that the full test accepts."""
import numpy as np

F = np.float32


def cylinders(rng, n):
    """Centres (internal frame, z forward) within a 60 degree view at 3..300 A, unit axes, half lengths, radii."""
    z = np.exp(rng.uniform(np.log(3.0), np.log(300.0), n))
    m = rng.uniform(-0.8, 0.8, (n, 2))
    hl = rng.uniform(0.02, 1.2, n)
    rb = rng.uniform(0.05, 0.5, n)
    z = np.maximum(z, 8.2 * (hl + rb))  # nearer ones take their bounding sphere's box
    A = rng.standard_normal((n, 3))
    A[: n // 8] = np.eye(3)[rng.integers(0, 3, n // 8)]  # axis-aligned ones among them
    A /= np.linalg.norm(A, axis=1, keepdims=True)
    return np.column_stack([m * z[:, None], z]), A, hl, rb


def test_reach_covers_every_point():
    """Points of the cylinder (rim, side, inside) project within the reach of entry_box, evaluated in FP32."""
    rng = np.random.default_rng(1)
    C, A, hl, rb = cylinders(rng, 200_000)
    f = 935.0
    c, a, h, r = (v.astype(F) for v in (C, A, hl, rb))
    for _ in range(12):
        w = np.cross(A, rng.standard_normal(A.shape))
        w *= (rb * rng.choice([1.0, 0.7], len(rb)) / np.linalg.norm(w, axis=1))[:, None]
        tau = hl * rng.choice([-1.0, 1.0, 0.3], len(hl))
        Q = C + tau[:, None] * A + w
        t = F(f) / (c[:, 2] - h * np.abs(a[:, 2]) - r) * F(1.001)
        for k in (0, 1):
            m = c[:, k] / c[:, 2]
            reach = t * (h * np.abs(a[:, k] - m * a[:, 2]) + r * (F(0.5) * m * m + F(1.0))) + F(0.01)
            off = f * np.abs(Q[:, k] / Q[:, 2] - C[:, k] / C[:, 2])
            assert np.all(off <= reach)


def hit_test(o, a, b, A, hl, rb, early):
    """cylinder_local in FP32, without contraction beyond its explicit multiply-adds (done in FP64 and rounded)."""
    def fma(x, y, z):
        return (x.astype(np.float64) * y.astype(np.float64) + z.astype(np.float64)).astype(F)

    one = np.ones_like(a)
    ua = fma(a, A[:, 0], fma(b, A[:, 1], A[:, 2]))
    oa = fma(o[:, 0], A[:, 0], fma(o[:, 1], A[:, 1], o[:, 2] * A[:, 2]))
    up = [fma(-ua, A[:, k], u) for k, u in enumerate((a, b, one))]
    op = [fma(-oa, A[:, k], o[:, k]) for k in range(3)]

    def dot(x, y):
        return fma(x[0], y[0], fma(x[1], y[1], x[2] * y[2]))

    a2, b2, opop = dot(up, up), dot(op, up), dot(op, op)
    c2 = fma(-rb, rb, opop)
    disc = fma(b2, b2, -a2 * c2)
    skip = (a2 > F(1e-12)) & (disc < F(-1e-5) * fma(b2, b2, a2 * (opop + rb * rb)))
    with np.errstate(all="ignore"):
        s1 = (-b2 - np.sqrt(np.maximum(disc, 0))) / a2
        best = np.where((a2 > F(1e-12)) & (disc >= 0) & (np.abs(fma(s1, ua, oa)) <= hl), s1, F(np.inf))
        for sign in (1, -1):
            sc = (F(sign) * hl - oa) / ua
            q = [fma(sc, up[k], op[k]) for k in range(3)]
            cap = (np.abs(ua) > F(1e-12)) & (dot(q, q) <= rb * rb) & (sc < best)
            best = np.where(cap, sc, best)
    hit = np.isfinite(best)
    return (hit & ~skip if early else hit), skip


def test_early_return_drops_no_hit():
    """Rays aimed at, along and just past the silhouette: the early return never fires where the full test hits, and
    fires for most of the rays that miss."""
    rng = np.random.default_rng(2)
    C, A, hl, rb = cylinders(rng, 400_000)
    n = len(hl)
    # aim: a point at distance rb (1 + e) from the axis, e from deep inside to far outside, many within 1e-6 of it
    e = np.concatenate([rng.uniform(-1, 3, n // 2), rng.normal(0, 1, n - n // 2) * 10.0 ** rng.uniform(-8, -2, n - n // 2)])
    w = np.cross(A, rng.standard_normal(A.shape))
    w *= (rb * (1 + e) / np.linalg.norm(w, axis=1))[:, None]
    Q = C + (hl * rng.uniform(-1.3, 1.3, n))[:, None] * A + w
    a, b = Q[:, 0] / Q[:, 2], Q[:, 1] / Q[:, 2]
    o = np.column_stack([a * C[:, 2] - C[:, 0], b * C[:, 2] - C[:, 1], np.zeros(n)])  # the ray at the centre's depth
    args = [v.astype(F) for v in (o, a, b, A, hl, rb)]
    full, skip = hit_test(*args, early=False)
    short, _ = hit_test(*args, early=True)
    assert np.array_equal(full, short)
    assert full.mean() > 0.2 and skip[~full].mean() > 0.3
