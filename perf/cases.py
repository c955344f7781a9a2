"""The work this renderer is used for, as cases to be timed.

Each case is one call of a user's program through the public API: a frame drawn into planes that the program keeps
(molecule viewing and trajectory playback), a trajectory batch, a differentiable soft-edge step, a solvent excluded
surface, an 8K image for print.  Sizes are those of the scenes module and of the benchmark (2,000 atoms at 256x256
through 1e8 atoms at 3840x2160), with odd sizes between them.  Scenes follow the same recipes as the scenes module
(uniform cubes, protein-like residue walks, whole-cell blobs), drawn with torch on the GPU so that 1e8 atoms take a
moment.

exact() computes a case's outputs in float64 with plain torch operations: a nearest-hit search over the candidate
pixels of every primitive, shading from the definitions in include/vtx.h, the soft compositor through autograd, and
the surface through a full distance transform and its own marching-cubes table.
"""
import math

import numpy as np
import torch

import paper_2501_12750_gb300 as vtx
from paper_2501_12750_gb300 import scenes

F64 = torch.float64
PROBE = 1.4


# ---------------------------------------------------------------------------------------------------- the cases --

def listed():
    return [
        # the smallest frame: a ligand-sized system in a 256x256 viewport, no ambient occlusion
        dict(name="frame_2k_256", kind="frame", layout="uniform", n=2000, width=256, height=256, style="plain"),
        # an illustration: solvent accessible surface, toon bands, outline, fog and a clip plane, odd sizes
        dict(name="frame_styled_30k", kind="frame", layout="protein", n=30011, width=1367, height=769, style="styled"),
        # the everyday view: one protein system in a full-HD viewport with ambient occlusion
        dict(name="frame_protein_1080p", kind="frame", layout="protein", n=100000, width=1920, height=1080,
             style="ssao"),
        # ball-and-stick (spheres and bond cylinders) seen from nearby
        dict(name="frame_sticks_60k", kind="frame", layout="protein", n=60000, width=1920, height=1080, style="bonds"),
        # flying into a cell: 1.1e7 atoms from 600 A outside, 4K, most of the screen covered
        dict(name="frame_cell_close_4k", kind="frame", layout="cell", n=11000000, width=3840, height=2160,
             style="ssao", close=True),
        # the whole-cell overview: 1e8 atoms, 4K
        dict(name="frame_cell_4k", kind="frame", layout="cell", n=100000000, width=3840, height=2160, style="ssao"),
        # a figure for print: 1.07e6 atoms at 8K, then RGBA8 with a transparent background
        dict(name="export_8k", kind="export", layout="cell", n=1070000, width=7680, height=4320, style="ssao"),
        # a trajectory: frames of uneven atom counts from four orbit cameras, one call
        dict(name="batch_500k_8x4", kind="batch", layout="protein", n=500000, frames=8, views=4, width=1280,
             height=720, style="ssao"),
        # structure-to-image fitting of a small ligand: one differentiable step, ragged image
        dict(name="soft_1k_2x200", kind="soft", layout="protein", n=1200, views=2, width=200, height=136),
        # the same for a 20,000-atom protein from 16 views
        dict(name="soft_20k_16x512", kind="soft", layout="protein", n=20000, views=16, width=512, height=512),
        # solvent excluded surface of a peptide
        dict(name="ses_1200", kind="ses", layout="protein", n=1200, spacing=0.6),
        # and of a whole protein system on a fine grid
        dict(name="ses_100k", kind="ses", layout="protein", n=100000, spacing=0.5),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["plain", "ssao", "cell", "styled", "bonds", "export", "batch", "soft", "ses"],
                       [1, 2, 2, 1, 1, 1, 1, 2, 2])[0]
    width = logint(240, 3840)
    height = max(160, min(2160, int(width * rng.uniform(0.5, 1.0))))
    c = dict(kind="frame", layout="protein", width=width, height=height, style=kind)
    if kind == "plain":
        c.update(layout=rng.choice(["uniform", "protein"]), n=logint(1500, 200000))
    elif kind == "ssao":
        c.update(n=logint(1500, 1000000))
    elif kind == "cell":
        c.update(layout="cell", style="ssao", n=logint(300000, 30000000), close=rng.random() < 0.4)
    elif kind in ("styled", "bonds"):
        c.update(n=logint(2000, 250000))
    elif kind == "export":
        w = logint(1920, 7680)
        c.update(kind="export", layout="cell", style="ssao", n=logint(100000, 4000000), width=w,
                 height=int(w * rng.uniform(0.5, 0.7)))
    elif kind == "batch":
        w = logint(200, 1280)
        c.update(kind="batch", style="ssao", n=logint(20000, 500000), frames=rng.randint(2, 8), views=rng.randint(1, 4),
                 width=w, height=int(w * rng.uniform(0.5, 1.0)))
    elif kind == "soft":
        w = logint(90, 512)
        c = dict(kind="soft", layout="protein", n=logint(300, 20000), views=rng.randint(1, 16), width=w,
                 height=int(w * rng.uniform(0.6, 1.0)))
    else:
        c = dict(kind="ses", layout="protein", n=logint(400, 110000), spacing=round(rng.uniform(0.5, 1.0), 3))
    return c


def work(case):
    n, kind = case["n"], case["kind"]
    if kind == "ses":
        # atoms read once, triangles written once: the surface of these systems has about 59 triangles an atom at
        # 0.5 A, and their number goes with 1 / spacing^2
        return {"bytes": 16.0 * n + 36.0 * 59.0 * n * (0.5 / case["spacing"]) ** 2, "flops": 0.0}
    pixels = float(case["width"] * case["height"])
    if kind == "soft":
        # planes written and upstream gradients read (5 floats a pixel each), atoms read twice, gradients written
        # once; 178 operations a composited term and about 33 terms an atom and view (vtx_soft_terms)
        return {"bytes": 40.0 * pixels * case["views"] + 48.0 * n, "flops": 178.0 * 33.0 * n * case["views"]}
    if kind == "batch":
        total = sum(_counts(case))
        return {"bytes": 16.0 * total + 36.0 * pixels * case["frames"] * case["views"], "flops": 0.0}
    # atom records read once; depth, id, normal, colour and occlusion planes written once (export: colour and id
    # read, RGBA8 written)
    extra = 20.0 * pixels if kind == "export" else 0.0
    return {"bytes": 16.0 * n + 36.0 * pixels + extra, "flops": 0.0}


# ----------------------------------------------------------------------------------------------------- scenes --

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _unit(gen, shape, dtype):
    v = torch.randn(shape + (3,), generator=gen, device=gen.device, dtype=dtype)
    return v / v.norm(dim=-1, keepdim=True)


def _jitter(gen, shape, radius, dtype):
    """Points uniform in a ball."""
    u = torch.rand(shape + (1,), generator=gen, device=gen.device, dtype=dtype)
    return _unit(gen, shape, dtype) * (radius * u ** (1.0 / 3.0))


def _walk(gen, chains, residues, start, inside):
    """Residue positions (chains, residues, 3) of 3.8 A step walks kept in by inside()."""
    steps = 3.8 * _unit(gen, (residues, chains), F64)
    p = start
    out = torch.empty((residues, chains, 3), dtype=F64, device=gen.device)
    for k in range(residues):
        if k:
            p = inside(p + steps[k])
        out[k] = p
    return out.transpose(0, 1)


def _protein(gen, n):
    """n atoms (n, 3): 300-residue chains reflected at the walls of a box of 1e5 atoms per (150 A)^3."""
    box = scenes.box_edge(n)
    chains = -(-n // 2400)

    def inside(p):
        return torch.where(p > box, 2.0 * box - p, torch.where(p < 0.0, -p, p))

    res = _walk(gen, chains, 300, box * torch.rand((chains, 3), generator=gen, device=gen.device, dtype=F64), inside)
    atoms = res[:, :, None, :] + _jitter(gen, (chains, 300, 8), 1.5, F64)
    return atoms.reshape(-1, 3)[:n], box


def _cell(gen, n):
    """n atoms in 5,000-atom blobs at the density of 20,000 blobs in a 12,000 A cube."""
    blobs = -(-n // 5000)
    edge = scenes.CELL_EDGE * (blobs / 20000.0) ** (1.0 / 3.0)
    centres = edge * torch.rand((blobs, 3), generator=gen, device=gen.device, dtype=F64)

    def inside(p):
        d = p.norm(dim=1, keepdim=True)
        return torch.where(d > 34.0, p * ((68.0 - d) / d.clamp(min=1e-30)), p)

    res = _walk(gen, blobs, 625, torch.zeros((blobs, 3), dtype=F64, device=gen.device), inside) + centres[:, None, :]
    atoms = torch.empty((blobs, 625, 8, 3), dtype=torch.float32, device=gen.device)
    for b in range(0, blobs, 2000):
        part = res[b:b + 2000]
        atoms[b:b + 2000] = part[:, :, None, :] + _jitter(gen, (part.shape[0], 625, 8), 1.5, torch.float32)
    return atoms.reshape(-1, 3)[:n], edge


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(seed)


def _atoms(case, gen):
    n = case["n"]
    if case["layout"] == "uniform":
        box = 40.0 * (n / 2000.0) ** (1.0 / 3.0)
        pos = box * torch.rand((n, 3), generator=gen, device=gen.device, dtype=F64)
    elif case["layout"] == "protein":
        pos, box = _protein(gen, n)
    else:
        pos, box = _cell(gen, n)
    cdf = torch.tensor(np.cumsum(scenes.ELEMENT_PROBS)[:-1], dtype=torch.float32, device=gen.device)
    elem = torch.bucketize(torch.rand(n, generator=gen, device=gen.device), cdf, right=True).to(torch.uint8)
    xyzr = torch.empty((n, 4), dtype=torch.float32, device=gen.device)
    xyzr[:, :3] = pos
    xyzr[:, 3] = torch.tensor(scenes.VDW_RADII, device=gen.device)[elem.long()]
    return xyzr, elem, box


def _bonds(xyzr):
    """Pairs i < j within 1.9 A among the atoms of one residue or of consecutive residues (8 atoms each)."""
    n = xyzr.shape[0] // 8 * 8
    p = xyzr[:n, :3].double().reshape(-1, 8, 3)
    first = 8 * torch.arange(p.shape[0], device=xyzr.device)

    def close(a, b, ia, ib, upper):
        d = (a[:, :, None, :] - b[:, None, :, :]).norm(dim=-1)
        ok = (d >= scenes.BOND_MIN) & (d < scenes.BOND_MAX)
        if upper:
            ok &= torch.ones(8, 8, dtype=torch.bool, device=a.device).triu(1)
        r, i, j = ok.nonzero(as_tuple=True)
        return torch.stack([ia[r] + i, ib[r] + j], 1)

    pairs = torch.cat([close(p, p, first, first, True), close(p[:-1], p[1:], first[:-1], first[1:], False)])
    order = torch.argsort(pairs[:, 0] * xyzr.shape[0] + pairs[:, 1])
    return pairs[order].to(torch.int32).contiguous()


def _cameras(case, box):
    w, h = case["width"], case["height"]
    centre = np.array([box / 2.0] * 3)
    if case["kind"] == "soft":  # orbit of azimuths and elevations
        views = [(90.0 * (k // 4), (-45.0, -15.0, 15.0, 45.0)[k % 4]) for k in range(16)]
        return [scenes.orbit_camera(centre, 3.0 * box, az, el, w, h) for az, el in views[:case["views"]]]
    if case["kind"] == "batch":
        return [scenes.orbit_camera(centre, 3.0 * box, 90.0 * k, 0.0, w, h) for k in range(case["views"])]
    if case["style"] == "bonds":  # near enough to tell balls from sticks
        return [scenes.look_at(centre + np.array([0.0, 0.0, 1.2 * box]), centre, w, h)]
    if case.get("close"):
        return [scenes.look_at(np.array([box / 2.0, box / 2.0, box + 600.0]), centre, w, h)]
    return [scenes.look_at(centre + np.array([0.0, 0.0, 3.0 * box]), centre, w, h)]


def _settings(case, box):
    style = case["style"]
    if style == "plain":
        return vtx.default_settings()
    if style == "ssao":
        return vtx.default_settings(ssao_kernel=scenes.ssao_kernel())
    if style == "bonds":
        return vtx.default_settings(ssao_kernel=scenes.ssao_kernel(), mode=vtx.MODE_BALL_AND_STICK)
    return vtx.default_settings(mode=vtx.MODE_SAS, shading=vtx.SHADE_TOON, outline_depth=2.0,
                                outline_color=(0.05, 0.05, 0.1), clip_plane=(0.0, 0.0, -1.0, 0.8 * box),
                                fog_near=2.5 * box, fog_far=3.6 * box, fog_density=0.6)


def _counts(case):
    """Atoms of each frame of a batch: frames of uneven size."""
    return [case["n"] - (37 * f * case["n"]) // 1000 for f in range(case["frames"])]


def _inputs(case, seed):
    """Everything but the renderer: the arrays, cameras and settings of a case."""
    gen = _generator(seed)
    xyzr, elem, box = _atoms(case, gen)
    s = dict(case=case, xyzr=xyzr, elem=elem)
    if case["kind"] == "ses":
        return s
    s["cams"] = _cameras(case, box)
    if case["kind"] == "soft":
        shape = (case["views"], case["height"], case["width"])
        s["upstream"] = [torch.randn(shape, generator=gen, device=gen.device) / (shape[1] * shape[2]),
                         0.01 * torch.randn(shape, generator=gen, device=gen.device) / (shape[1] * shape[2]),
                         torch.randn((shape[0], 3) + shape[1:], generator=gen, device=gen.device)
                         / (shape[1] * shape[2])]
        return s
    s["settings"] = _settings(case, box)
    if case["kind"] == "batch":  # a Gaussian walk of every atom, 0.3 A a frame and coordinate
        step = torch.zeros((case["frames"], case["n"], 4), device=gen.device)
        step[1:, :, :3] = 0.3 * torch.randn((case["frames"] - 1, case["n"], 3), generator=gen, device=gen.device)
        s["frames"] = (xyzr[None] + step.double().cumsum(0)).float().contiguous()
        s["counts"] = _counts(case)
    s["bonds"] = _bonds(xyzr) if case["style"] == "bonds" else None
    return s


def _mesh_buffer(case, dtype, device):
    """The program's own vertex buffer, which the mesh of each pass is copied into."""
    room = int(140 * case["n"] * (0.5 / case["spacing"]) ** 2) + 4096
    return torch.zeros((room, 3, 3), dtype=dtype, device=device)


def prepare(case, seed):
    """Inputs, a renderer and the planes that a program keeps.  Asynchronous frames need the arena sized, which
    a program does with one synchronising frame."""
    s = _inputs(case, seed)
    s["renderer"] = r = vtx.Renderer()
    if case["kind"] == "ses":
        s["mesh"] = _mesh_buffer(case, torch.float32, s["xyzr"].device)
        return s
    if case["kind"] == "soft":
        s["xyzr"].requires_grad_(True)
        return s
    flags, s["settings"].flags = s["settings"].flags, vtx.FLAG_SYNC
    if case["kind"] == "batch":
        r.upload_atoms(s["frames"][0], s["elem"])
        s["out"] = r.alloc_outputs(case["width"], case["height"], case["frames"] * case["views"])
        r.render_batch(s["frames"], s["counts"], s["cams"], s["settings"], out=s["out"])
    else:
        r.upload_atoms(s["xyzr"], s["elem"])
        if s["bonds"] is not None:
            r.upload_bonds(s["bonds"])
        r.set_camera(s["cams"][0])
        s["out"] = r.alloc_outputs(case["width"], case["height"])
        r.render_frame(s["settings"], out=s["out"])
        if case["kind"] == "export":
            s["rgba"] = torch.empty((case["height"], case["width"], 4), dtype=torch.uint8, device="cuda")
    s["settings"].flags = flags
    return s


def run(s):
    case, r = s["case"], s["renderer"]
    if case["kind"] == "soft":
        planes = vtx.SoftRender.apply(s["xyzr"], r, s["cams"], 0.5)
        grad, = torch.autograd.grad(planes, s["xyzr"], s["upstream"])
        return dict(coverage=planes[0].detach(), depth=planes[1].detach(), normal=planes[2].detach(), grad=grad)
    if case["kind"] == "ses":
        mesh = r.ses_mesh(s["xyzr"], r.ses_fit_grid(s["xyzr"], probe=PROBE, spacing=case["spacing"]))
        s["mesh"][:mesh["n"]] = mesh["tris"]
        return dict(tris=s["mesh"], n=mesh["n"])
    if case["kind"] == "batch":
        return r.render_batch(s["frames"], s["counts"], s["cams"], s["settings"], out=s["out"])
    out = r.render_frame(s["settings"], out=s["out"])
    if case["kind"] == "export":
        return dict(out, rgba=r.export_rgba8(out, background_alpha=0.0, rgba=s["rgba"]))
    return out


# ------------------------------------------------------------------------------------------ exact: hard frames --

class _View:
    """A camera in float64: x right, y up, z forward, rays (a, b, 1)."""

    def __init__(self, cam, device):
        def t(v):
            return torch.tensor(np.asarray(v, np.float64), device=device)

        self.eye, self.basis = t(cam.eye), torch.stack([t(cam.right), t(cam.up), t(cam.forward)])
        self.w, self.h = cam.width, cam.height
        self.f = cam.height / (2.0 * float(cam.tan_half_fovy))
        self.near = float(cam.znear)

    def points(self, xyz):
        return (xyz.double() - self.eye) @ self.basis.T

    def ray(self, pix):
        px, py = pix % self.w, torch.div(pix, self.w, rounding_mode="floor")
        a, b = (px + 0.5 - 0.5 * self.w) / self.f, (0.5 * self.h - py - 0.5) / self.f
        return a, b, a * a + b * b + 1.0

    def boxes(self, c, r):
        """Candidate pixel boxes of spheres (view centre c, radius r), conservative; empty ones have zero width."""
        z = c[:, 2]
        ok = (z > 1.05 * r) & (z + r > self.near)
        rho = torch.where(ok, r / z, torch.zeros_like(z))
        out = []
        for k, size in ((0, self.w), (1, self.h)):
            m = torch.where(ok, c[:, k] / z, torch.zeros_like(z))
            reach = self.f * rho / (1.0 - rho * rho) * (m.abs() * rho + (1.0 + m * m).sqrt()) + 0.01
            u = 0.5 * size + (self.f if k == 0 else -self.f) * m - 0.5
            lo, hi = (u - reach).ceil().clamp(min=0), (u + reach).floor().clamp(max=size - 1)
            out += [lo.long(), torch.where(ok, (hi - lo + 1).clamp(min=0), torch.zeros_like(lo)).long()]
        return out


def _pairs(view, centre, radius, most=1 << 24):
    """(primitive, pixel) index pairs of all candidate boxes, in chunks."""
    x0, w, y0, h = view.boxes(centre, radius)
    live = ((w > 0) & (h > 0)).nonzero().squeeze(1)
    end = (w[live] * h[live]).cumsum(0)
    i = 0
    while i < len(live):
        base = int(end[i - 1]) if i else 0
        j = max(i + 1, int(torch.searchsorted(end, base + most, right=True)))
        part = live[i:j]
        count = w[part] * h[part]
        who = torch.repeat_interleave(part, count)
        k = torch.arange(len(who), device=who.device) - torch.repeat_interleave(count.cumsum(0) - count, count)
        yield who, (y0[who] + k // w[who]) * view.w + x0[who] + k % w[who]
        i = j


def _hit_sphere(view, pix, c, r):
    """Entry depth (inf: no hit) and normal (view frame, z forward)."""
    a, b, uu = view.ray(pix)
    u = torch.stack([a, b, torch.ones_like(a)], 1)
    tc = (u * c).sum(1) / uu
    disc = r * r - (c - tc[:, None] * u).square().sum(1)
    t = tc - (disc.clamp(min=0.0) / uu).sqrt()
    return torch.where((disc >= 0.0) & (t >= view.near), t, math.inf), (t[:, None] * u - c) / r[:, None]


def _hit_cylinder(view, pix, A, B, rad):
    """Entry depth, normal and axial position (relative to the middle) of a capped cylinder from A to B."""
    a, b, _ = view.ray(pix)
    u = torch.stack([a, b, torch.ones_like(a)], 1)
    mid, axis = 0.5 * (A + B), B - A
    half = 0.5 * axis.norm(dim=1)
    axis = axis / (2.0 * half)[:, None]
    o = mid[:, 2:3] * u - mid  # the ray at the middle's depth
    ua, oa = (u * axis).sum(1), (o * axis).sum(1)
    up, op = u - ua[:, None] * axis, o - oa[:, None] * axis
    qa, qb, qc = up.square().sum(1), (up * op).sum(1), op.square().sum(1) - rad * rad
    disc = qb * qb - qa * qc
    s = (-qb - disc.clamp(min=0.0).sqrt()) / qa.clamp(min=1e-300)
    best = torch.where((disc >= 0.0) & (qa > 1e-24) & ((oa + s * ua).abs() <= half), s, math.inf)
    normal = (op + s[:, None] * up) / rad
    for sign in (1.0, -1.0):
        s = (sign * half - oa) / torch.where(ua == 0.0, torch.ones_like(ua), ua)
        cap = (ua != 0.0) & ((op + s[:, None] * up).square().sum(1) <= rad * rad) & (s < best)
        best = torch.where(cap, s, best)
        normal = torch.where(cap[:, None], sign * axis, normal)
    t = mid[:, 2] + best
    return torch.where(t >= view.near, t, math.inf), normal, oa + best * ua


def _radii(xyzr, s):
    if s.mode == vtx.MODE_BALL_AND_STICK:
        return torch.full_like(xyzr[:, 3], s.ball_radius)
    return xyzr[:, 3] + s.probe_radius if s.mode == vtx.MODE_SAS else xyzr[:, 3]  # stored radii are float32 sums


def _exact_frame(xyzr, elem, bonds, cam, s):
    """depth, id, normal, rgb and ao planes of one image in float64 (id: int32)."""
    dev = xyzr.device
    view = _View(cam, dev)
    n, pixels = xyzr.shape[0], cam.width * cam.height
    inf = float("inf")
    depth = torch.full((pixels,), inf, dtype=F64, device=dev)
    ident = torch.full((pixels,), 1 << 40, dtype=torch.int64, device=dev)
    plane = torch.tensor(list(s.clip_plane), dtype=F64, device=dev)
    chunk = 1 << 22

    def sphere_hits():
        for a0 in range(0, n, chunk):
            part = xyzr[a0:a0 + chunk]
            c, r = view.points(part[:, :3]), _radii(part, s).double()
            if bool(plane[:3].any()):
                kept = part[:, :3].double() @ plane[:3] + plane[3] >= 0.0
                r = torch.where(kept, r, torch.full_like(r, -1.0))
                c = torch.where(kept[:, None], c, torch.full_like(c, -1.0))
            for who, pix in _pairs(view, c, r):
                yield a0 + who, pix, _hit_sphere(view, pix, c[who], r[who])[0]

    def bond_hits():
        A, B = (view.points(xyzr[bonds[:, k].long(), :3]) for k in (0, 1))
        bound = (0.25 * (B - A).square().sum(1) + s.bond_radius ** 2).sqrt()
        for who, pix in _pairs(view, 0.5 * (A + B), bound, 1 << 22):
            yield n + who, pix, _hit_cylinder(view, pix, A[who], B[who], float(s.bond_radius))[0]

    for hits in (sphere_hits, bond_hits) if bonds is not None else (sphere_hits,):
        for who, pix, t in hits():
            depth.scatter_reduce_(0, pix, t, "amin")
    for hits in (sphere_hits, bond_hits) if bonds is not None else (sphere_hits,):
        for who, pix, t in hits():
            won = (t == depth[pix]) & (t < inf)
            ident.scatter_reduce_(0, pix[won], who[won], "amin")

    planes = dict(depth=depth.clone(), id=torch.full((pixels,), -1, dtype=torch.int32, device=dev),
                  normal=torch.zeros((3, pixels), dtype=F64, device=dev),
                  rgb=torch.tensor(list(s.background), dtype=F64, device=dev)[:, None].repeat(1, pixels),
                  ao=torch.ones(pixels, dtype=F64, device=dev))
    for pix in (depth < inf).nonzero().squeeze(1).split(1 << 20):
        _shade(view, s, xyzr, elem, bonds, depth, ident, pix, planes)
    shape = (cam.height, cam.width)
    return {k: v.reshape(v.shape[:-1] + shape) for k, v in planes.items()}


def _shade(view, s, xyzr, elem, bonds, depth, ident, pix, planes):
    dev, n = xyzr.device, xyzr.shape[0]
    who, t = ident[pix], depth[pix]
    atom = who.clamp(max=n - 1)
    c = view.points(xyzr[atom, :3])
    normal = _hit_sphere(view, pix, c, _radii(xyzr[atom], s).double())[1]
    if bonds is not None:
        stick = (who >= n).nonzero().squeeze(1)
        pair = bonds[who[stick] - n].long()
        A, B = (view.points(xyzr[pair[:, k], :3]) for k in (0, 1))
        _, cyl, axial = _hit_cylinder(view, pix[stick], A, B, float(s.bond_radius))
        normal[stick] = cyl
        atom[stick] = torch.where(axial <= 0.0, pair[:, 0], pair[:, 1])
    nrm = normal * torch.tensor([1.0, 1.0, -1.0], dtype=F64, device=dev)  # z toward the viewer
    a, b, uu = view.ray(pix)
    ray = torch.stack([a, b, -torch.ones_like(a)], 1)
    albedo = torch.tensor(scenes.PALETTE, dtype=F64, device=dev)[elem[atom].long()]
    light = torch.tensor(list(s.light_dir), dtype=F64, device=dev)
    light = light / light.norm()
    nl = nrm @ light
    if s.shading == vtx.SHADE_TOON:
        bands = float(s.toon_levels)
        nl = (nl.clamp(min=0.0) * bands).floor().clamp(max=bands - 1.0) / (bands - 1.0)
        rgb = (albedo * (s.ka + s.kd * nl)[:, None]).clamp(max=1.0)
    else:
        half = light - ray / uu.sqrt()[:, None]
        nh = (nrm * half).sum(1) / half.norm(dim=1)
        spec = torch.where(nl > 0.0, s.ks * nh.clamp(min=0.0) ** s.shininess, torch.zeros_like(nl))
        rgb = (albedo * (s.ka + s.kd * nl.clamp(min=0.0))[:, None] + spec[:, None]).clamp(0.0, 1.0)

    def at(x, y):
        ok = (x >= 0) & (y >= 0) & (x < view.w) & (y < view.h)
        z = depth[torch.where(ok, y * view.w + x, torch.zeros_like(x))]
        return ok, z

    ao = torch.ones_like(t)
    if s.ssao_samples:
        up = torch.zeros_like(nrm)
        steep = nrm[:, 1].abs() > 0.9
        up[:, 0], up[:, 1] = steep.double(), (~steep).double()
        tangent = torch.linalg.cross(nrm, up)
        tangent = tangent / tangent.norm(dim=1, keepdim=True)
        other = torch.linalg.cross(nrm, tangent)
        blocked = torch.zeros_like(t)
        for j in range(s.ssao_samples):
            k = list(s.ssao_kernel[j])
            off = s.ssao_radius * (k[0] * tangent + k[1] * other + k[2] * nrm)
            p = t[:, None] * ray + off
            z = -p[:, 2]
            front = z > 0.0
            zs = torch.where(front, z, torch.ones_like(z))
            # the offset from the pixel's own centre, so that a small one is not lost in the coordinate
            dx = view.f * (off[:, 0] + a * off[:, 2]) / zs
            dy = -view.f * (off[:, 1] + b * off[:, 2]) / zs
            x = pix % view.w + (0.5 + dx).floor().long()
            y = torch.div(pix, view.w, rounding_mode="floor") + (0.5 + dy).floor().long()
            ok, zf = at(x, y)
            dz = zf - t
            hit = front & ok & torch.isfinite(zf) & (dz <= -off[:, 2] - s.ssao_bias)
            blocked += torch.where(hit, (s.ssao_radius / dz.abs().clamp(min=1e-300)).clamp(max=1.0),
                                   torch.zeros_like(dz))
        ao = 1.0 - blocked / s.ssao_samples
        rgb = rgb * ao[:, None]
    if s.outline_depth > 0.0:
        edge = torch.zeros_like(t, dtype=torch.bool)
        x, y = pix % view.w, torch.div(pix, view.w, rounding_mode="floor")
        for dx, dy in ((-1, 0), (1, 0), (0, -1), (0, 1)):
            ok, z = at(x + dx, y + dy)
            edge |= ok & (z - t > s.outline_depth)
        rgb = torch.where(edge[:, None], torch.tensor(list(s.outline_color), dtype=F64, device=dev), rgb)
    if s.fog_density > 0.0:
        fog = s.fog_density * ((t - s.fog_near) / (s.fog_far - s.fog_near)).clamp(0.0, 1.0)
        rgb = rgb + fog[:, None] * (torch.tensor(list(s.background), dtype=F64, device=dev) - rgb)
    planes["id"][pix] = who.to(torch.int32)
    planes["normal"][:, pix] = nrm.T
    planes["rgb"][:, pix] = rgb.T
    planes["ao"][pix] = ao


# ------------------------------------------------------------------------------------------------- exact: soft --

def _exact_soft(s, sigma=0.5):
    x = s["xyzr"].detach().double().requires_grad_(True)
    total, cov, dep, nrm = torch.zeros_like(x), [], [], []
    for k, cam in enumerate(s["cams"]):
        view = _View(cam, x.device)
        with torch.no_grad():
            c, r = view.points(x[:, :3]), x[:, 3]
            order = torch.argsort(c[:, 2], stable=True)  # centre depth, then id
            order = order[c[order, 2] > view.near]
            c, r = c[order], r[order]
            who, pix = [], []
            for w, p in _pairs(view, c, r + 4.2 * c[:, 2] / view.f, 1 << 22):
                a, b, uu = view.ray(p)
                u = torch.stack([a, b, torch.ones_like(a)], 1)
                rho2 = (c[w] - ((u * c[w]).sum(1) / uu)[:, None] * u).square().sum(1)
                keep = (r[w] - (rho2 + 1e-12).sqrt()) * view.f / c[w, 2] >= -4.0
                who.append(w[keep])
                pix.append(p[keep])
            who, pix = torch.cat(who), torch.cat(pix)
            by = torch.argsort(pix, stable=True)
            who, pix = order[who[by]], pix[by]
            at, count = torch.unique_consecutive(pix, return_counts=True)
        A, D = (torch.zeros(view.w * view.h, dtype=F64, device=x.device) for _ in range(2))
        N = torch.zeros((3, view.w * view.h), dtype=F64, device=x.device)
        g = [u[k].reshape(-1, view.w * view.h).double() for u in s["upstream"]]
        start = count.cumsum(0) - count
        for p0 in range(0, len(at), 8192):
            rows = slice(p0, min(p0 + 8192, len(at)))
            rank = torch.arange(int(count[rows].max()), device=x.device)
            live = rank[None, :] < count[rows, None]
            idx = who[torch.where(live, start[rows, None] + rank, start[rows, None])]
            a, b, uu = (v[:, None] for v in view.ray(at[rows]))
            p = (x[idx, :3] - view.eye) @ view.basis.T
            r = x[idx, 3]
            u = torch.stack([a, b, torch.ones_like(a)], 2)
            tc = (u * p).sum(2) / uu
            rho2 = (p - tc[..., None] * u).square().sum(2)
            delta = (r - (rho2 + 1e-12).sqrt()) * view.f / p[..., 2]
            alpha = torch.sigmoid(delta / sigma).clamp(max=0.99) * live
            eta = 0.05 * r
            t = tc - (((r * r - rho2).clamp(min=0.0) + eta * eta).sqrt() - eta) / uu.sqrt()
            n = (t[..., None] * u - p) / r[..., None]
            left = torch.log1p(-alpha).cumsum(1) - torch.log1p(-alpha)
            weight = alpha * left.exp()
            weight = weight * (left.detach().exp() >= 1e-4)  # nothing after the transmittance falls below 1e-4
            planes = [weight.sum(1), (weight * t).sum(1), (weight[..., None] * n).sum(1)]
            planes[2] = planes[2] * torch.tensor([1.0, 1.0, -1.0], dtype=F64, device=x.device)
            pixels = at[rows]
            loss = (planes[0] * g[0][0, pixels]).sum() + (planes[1] * g[1][0, pixels]).sum() + \
                (planes[2] * g[2][:, pixels].T).sum()
            total += torch.autograd.grad(loss, x)[0]
            A[pixels], D[pixels], N[:, pixels] = planes[0].detach(), planes[1].detach(), planes[2].detach().T
        shape = (view.h, view.w)
        cov.append(A.reshape(shape))
        dep.append(D.reshape(shape))
        nrm.append(N.reshape((3,) + shape))
    return dict(coverage=torch.stack(cov), depth=torch.stack(dep), normal=torch.stack(nrm), grad=total)


# -------------------------------------------------------------------------------------------------- exact: SES --

CORNERS = np.array([(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)])
EDGES = [(0, 1), (1, 2), (2, 3), (3, 0), (4, 5), (5, 6), (6, 7), (7, 4), (0, 4), (1, 5), (2, 6), (3, 7)]
FACES = [((0, 3, 2, 1), (0, 0, -1)), ((4, 5, 6, 7), (0, 0, 1)), ((0, 1, 5, 4), (0, -1, 0)), ((2, 3, 7, 6), (0, 1, 0)),
         ((0, 4, 7, 3), (-1, 0, 0)), ((1, 2, 6, 5), (1, 0, 0))]


def _loops(case):
    """Loops of crossing edges of a cell, counter-clockwise about the outward normal, each from its smallest edge."""
    edge_of = {frozenset(e): k for k, e in enumerate(EDGES)}
    middle = [CORNERS[list(e)].mean(0) for e in EDGES]
    after = {}
    for ring, normal in FACES:
        inside = [c for c in ring if case >> c & 1]
        crossing = [edge_of[frozenset((ring[q], ring[(q + 1) % 4]))] for q in range(4)
                    if (case >> ring[q] & 1) != (case >> ring[(q + 1) % 4] & 1)]
        cuts = [(crossing, inside)] if len(crossing) == 2 else []
        if len(crossing) == 4:  # every inside corner is cut off on its own
            cuts = [([edge_of[frozenset((ring[q - 1], ring[q]))], edge_of[frozenset((ring[q], ring[(q + 1) % 4]))]],
                     [ring[q]]) for q in range(4) if case >> ring[q] & 1]
        for (e0, e1), corners in cuts:
            away = 0.5 * (middle[e0] + middle[e1]) - CORNERS[corners].mean(0)
            along = np.dot(middle[e1] - middle[e0], np.cross(away, normal))
            after.update({e0: e1} if along > 0 else {e1: e0})
    loops = []
    while after:
        loop = [min(after)]
        while loop[-1] in after:
            loop.append(after.pop(loop[-1]))
        loops.append(loop[:-1])
    return loops


def _triangle_table():
    """Per case: triangle count, vertices (0..11 an edge, 12 + l the mean of loop l), and the weights of the means."""
    count, verts, mean = np.zeros(256, np.int64), np.zeros((256, 12, 3), np.int64), np.zeros((256, 4, 12))
    for case in range(256):
        tris = []
        for q, loop in enumerate(_loops(case)):
            mean[case, q, loop] = 1.0 / len(loop)
            tris += [loop] if len(loop) == 3 else [(12 + q, e, loop[(k + 1) % len(loop)]) for k, e in enumerate(loop)]
        count[case] = len(tris)
        verts[case, :len(tris)] = np.array(tris).reshape(-1, 3)
    return count, verts, mean


def _exact_ses(x, h32):
    dev = x.device
    h, p = float(np.float32(h32)), float(np.float32(PROBE))
    reach = x[:, 3:4] + torch.tensor(PROBE, dtype=torch.float32, device=dev)  # the fitted grid is a float32 record
    lo, hi = (x[:, :3] - reach).amin(0).double(), (x[:, :3] + reach).amax(0).double()
    origin = (lo - 2.0 * h).float().double()
    dims = [int(v) for v in (((hi - lo) / h).floor() + 6.0).tolist()]
    nx, ny, nz = dims
    window = math.ceil(p / h) + 1

    # points inside a solvent accessible sphere
    sas = torch.zeros(nx * ny * nz, dtype=torch.bool, device=dev)
    c, r2 = x[:, :3].double(), (x[:, 3].double() + p) ** 2
    base = ((c - origin) / h).floor().long()
    m = math.ceil((float(x[:, 3].max()) + p) / h)
    along = [[(origin[d] + h * (base[:, d] + k).double() - c[:, d]).square() for k in range(-m, m + 2)] for d in range(3)]
    for dz in range(-m, m + 2):
        for dy in range(-m, m + 2):
            row = ((base[:, 2] + dz) * ny + base[:, 1] + dy) * nx + base[:, 0]
            fits = (base[:, 1] + dy >= 0) & (base[:, 1] + dy < ny) & (base[:, 2] + dz >= 0) & (base[:, 2] + dz < nz)
            for dx in range(-m, m + 2):
                d2 = along[0][dx + m] + along[1][dy + m] + along[2][dz + m]
                ok = (d2 < r2) & fits & (base[:, 0] + dx >= 0) & (base[:, 0] + dx < nx)
                sas[(row + dx)[ok]] = True

    # squared distance (grid units) to the nearest point outside, within the window
    far = 1 << 24
    dist = torch.where(sas.reshape(nz, ny, nx), far, 0).to(torch.int32)
    for axis in (2, 1, 0):
        best = dist.clone()
        for k in range(1, window + 1):
            for shift in (k, -k):
                moved = torch.full_like(dist, far)
                size = dist.shape[axis] - k
                if size > 0:
                    src, dst = (0, k) if shift > 0 else (k, 0)
                    moved.narrow(axis, dst, size).copy_(dist.narrow(axis, src, size))
                best = torch.minimum(best, moved + k * k)
        dist = best
    dist = dist.clamp(max=window * window + 1)
    inside = (dist >= 1) & (dist.double() * (h * h) >= p * p)

    cells = torch.zeros((nz - 1, ny - 1, nx - 1), dtype=torch.int64, device=dev)
    for k, (i, j, l) in enumerate(CORNERS):
        cells |= inside[l:l + nz - 1, j:j + ny - 1, i:i + nx - 1].long() << k
    count, verts, mean = (torch.from_numpy(v).to(dev) for v in _triangle_table())
    cells = cells.reshape(-1)
    active = (count[cells] > 0).nonzero().squeeze(1)
    field = dist.reshape(-1).double().sqrt() * h - p
    out = []
    for cell in active.split(1 << 19):
        case = cells[cell]
        at = torch.stack([cell % (nx - 1), (cell // (nx - 1)) % (ny - 1), cell // ((nx - 1) * (ny - 1))], 1)
        corner = at[:, None, :] + torch.from_numpy(CORNERS).to(dev)
        value = field[(corner[..., 2] * ny + corner[..., 1]) * nx + corner[..., 0]]
        place = origin + h * corner.double()
        e0, e1 = ([e[k] for e in EDGES] for k in (0, 1))
        f0, f1 = value[:, e0], value[:, e1]
        t = torch.where(f0 == f1, 0.5, f0 / torch.where(f0 == f1, 1.0, f0 - f1)).clamp(0.0, 1.0)[..., None]
        points = place[:, e0] + t * (place[:, e1] - place[:, e0])
        points = torch.cat([points, mean[case] @ points], 1)
        which = torch.repeat_interleave(torch.arange(len(cell), device=dev), count[case])
        first = torch.repeat_interleave(count[case].cumsum(0) - count[case], count[case])
        corner_of = verts[case[which], torch.arange(len(which), device=dev) - first]
        out.append(points[which[:, None], corner_of])
    return torch.cat(out)


# ------------------------------------------------------------------------------------------------------- exact --

def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "soft":
        return _exact_soft(s)
    if case["kind"] == "ses":
        tris = _exact_ses(s["xyzr"], case["spacing"])
        mesh = _mesh_buffer(case, F64, tris.device)
        mesh[:len(tris)] = tris
        return dict(tris=mesh, n=len(tris))
    if case["kind"] == "batch":
        images = [_exact_frame(s["frames"][f, :n], s["elem"], None, cam, s["settings"])
                  for f, n in enumerate(s["counts"]) for cam in s["cams"]]
        planes = {k: torch.stack([i[k] for i in images]) for k in images[0]}
        return planes if len(images) > 1 else images[0]
    out = _exact_frame(s["xyzr"], s["elem"], s["bonds"], s["cams"][0], s["settings"])
    if case["kind"] == "export":
        rgb = (out["rgb"].clamp(0.0, 1.0) * 255.0).round()
        alpha = torch.where(out["id"] >= 0, 255.0, 0.0)[None]
        out["rgba"] = torch.cat([rgb, alpha]).permute(1, 2, 0).to(torch.uint8)
    return out
