"""Performance cases: what users of the projectors have them do, at the sizes they do it.

A case is one scan geometry (fan beam, circular cone beam with a flat or a
curved detector, non-circular "saddle" cone beam with per-view pose jitter), a
volume and detector size, a storage type, and one operation:

  pair   a forward projection of a volume and a backprojection of a sinogram,
         the two calls an iterative method alternates;
  grad   the least-squares data term of a volume and its gradient through
         autograd (training and gradient-based reconstruction);
  mbir   a few least-squares gradient steps from zero (what the server runs);
  fbp    filtered backprojection of a sinogram (ramp filter, recon-mode back).

The fields of view, distances and detector extents are those of the four
workloads of this repository; sizes sample the same field of view.  `exact`
restates the projectors with plain torch in 64 bits from their definitions.
"""
import math

import numpy as np
import torch

import paper_2503_16741_gb300 as ct
from paper_2503_16741_gb300 import mbir

# field of view x, y, z; detector extent u, v; SAD; SDD (mm)
SCANS = {
    "fan": dict(fov=(128.0, 128.0, 1.0), det=(307.2, 1.0), sad=500.0, sdd=1000.0),
    "circ": dict(fov=(128.0, 128.0, 128.0), det=(409.6, 307.2), sad=785.0, sdd=1085.0),
    "curved": dict(fov=(409.6, 409.6, 32.0), det=(888.0, 64.0), sad=595.0, sdd=1085.6),
    "saddle": dict(fov=(204.8, 204.8, 204.8), det=(409.6, 409.6), sad=785.0, sdd=1200.0),
}
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BODIES = 8  # ellipsoids per phantom


def _case(name, scan, op, projector, n, nz, nu, nv, views, dtype="f32", batch=1, adjoint="", steps=0):
    return dict(name=name, scan=scan, op=op, projector=projector, adjoint=adjoint or projector, n=n, nz=nz, nu=nu,
                nv=nv, views=views, dtype=dtype, batch=batch, steps=steps)


def listed():
    return [
        # a single small fan-beam image, the unmatched pair of classic toolboxes: latency
        _case("fan_ray_voxel_128", "fan", "pair", "ray", 128, 1, 256, 1, 180, adjoint="voxel"),
        # a fan-beam slice of clinical size, analytic reconstruction
        _case("fan_fbp_512", "fan", "fbp", "voxel", 512, 1, 1024, 1, 720),
        # a small batch of odd-sized slices in a training step
        _case("fan_sf_grad_301", "fan", "grad", "sf", 301, 1, 603, 1, 217, batch=2),
        # the smallest served solve: a short reconstruction of a small volume
        _case("circ_dd_mbir_64", "circ", "mbir", "dd", 64, 64, 128, 96, 90, steps=3),
        # the headline workload: SF forward and back of a 256^3 volume
        _case("circ_sf_256", "circ", "pair", "sf", 256, 256, 512, 384, 360),
        # an odd-sized request in half storage
        _case("circ_dd_f16_183", "circ", "pair", "dd", 183, 157, 379, 277, 231, dtype="f16"),
        # analytic cone-beam reconstruction of the headline scan
        _case("circ_fbp_256", "circ", "fbp", "voxel", 256, 256, 512, 384, 360),
        # exact line integrals and their adjoint
        _case("circ_ray_128", "circ", "pair", "ray", 128, 128, 256, 192, 180),
        # large cone angles: trapezoid-trapezoid footprints, two channels in bfloat16
        _case("circ_sftt_96", "circ", "pair", "sftt", 96, 96, 192, 144, 120, dtype="bf16", batch=2),
        # the multi-row clinical scanner: one gradient of the data term, the largest case
        _case("curved_dd_grad_512", "curved", "grad", "dd", 512, 128, 888, 64, 984),
        # the non-circular scan in half storage
        _case("saddle_sf_f16_192", "saddle", "pair", "sf", 192, 192, 384, 384, 250, dtype="f16"),
        # a small non-circular request
        _case("saddle_dd_64", "saddle", "pair", "dd", 64, 64, 128, 128, 90),
    ]


#: what a drawn case may cost; curved_dd_grad_512, the largest listed one, costs 66e9
MOST = 40e9


def _passes(c):
    return {"pair": 2, "grad": 2, "fbp": 1}.get(c["op"], 2 * c["steps"])


def _updates(c):
    """(voxel, view) pairs of one pass."""
    return _passes(c) * c["batch"] * c["n"] * c["n"] * c["nz"] * c["views"]


def _cost(c):
    heavy = 12 if c["scan"] == "saddle" else 2.5 if c["projector"] in ("ray", "sftt", "voxel") else 1
    return heavy * _updates(c)


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    scan = rng.choice(["fan", "circ", "circ", "curved", "saddle"])
    lo, hi = {"fan": (96, 1024), "circ": (48, 272), "curved": (96, 512), "saddle": (40, 208)}[scan]
    n = log(lo, hi)
    if rng.random() < 0.5:  # half of the requests come in round sizes
        n = max(lo, n // 16 * 16)
    op = rng.choice(["pair", "pair", "pair", "grad", "mbir", "fbp"])
    if op == "fbp":
        projector = rng.choice(["voxel", "voxel", "dd", "sf"]) if scan != "saddle" else "voxel"
    elif op == "pair":
        projector = rng.choice(["sf", "dd", "sf", "dd", "ray", "voxel"] + (["sftt"] if scan == "circ" else []))
        if scan == "saddle" and projector in ("ray", "voxel"):
            projector = "sf"
    else:
        projector = rng.choice(["sf", "dd"])
    adjoint = "voxel" if op == "pair" and projector == "ray" and rng.random() < 0.5 else projector
    dtype = "f32" if op == "grad" else rng.choice(["f32", "f32", "f32", "f16", "bf16"])
    batch = rng.choice([1, 1, 1, 2, 3]) if scan == "fan" or n <= 128 else 1
    nz = {"fan": 1, "circ": round(n * rng.uniform(0.5, 1.05)), "curved": round(n * rng.uniform(0.18, 0.3)),
          "saddle": round(n * rng.uniform(0.7, 1.0))}[scan]
    nu = round(n * rng.uniform(1.6, 2.1))
    nv = {"fan": 1, "circ": round(n * rng.uniform(1.0, 1.55)), "curved": rng.choice([16, 32, 40, 64, 64, 96]),
          "saddle": round(n * rng.uniform(1.5, 2.0))}[scan]
    c = dict(scan=scan, op=op, projector=projector, adjoint=adjoint, n=n, nz=nz, nu=nu, nv=nv, views=log(60, 984),
             dtype=dtype, batch=batch, steps=rng.choice([2, 3]) if op == "mbir" else 0)
    while _cost(c) > MOST and c["views"] > 45:
        c["views"] = max(45, c["views"] * 3 // 4)
    return c


# ------------------------------------------------------------ scan geometry
def _params(c):
    """The per-view scan parameters a user gives (angles in radians, mm)."""
    s, nv = SCANS[c["scan"]], c["views"]
    p = dict(theta=0.3 + 2 * math.pi * np.arange(nv) / nv, sad=s["sad"], sdd=s["sdd"])
    if c["scan"] == "saddle":
        rng = np.random.default_rng(0)
        deg = math.pi / 180
        jit = lambda w: rng.uniform(-w, w, nv)  # noqa: E731
        p["phi"] = 5 * deg * np.cos(2 * p["theta"]) + jit(0.5 * deg)
        p["theta"] = p["theta"] + jit(0.5 * deg)
        p["psi"] = jit(0.5 * deg)
        for k in ("x_src", "z_src", "u_ofst", "v_ofst"):
            p[k] = jit(2.0)
    return p


def _steps(c):
    s = SCANS[c["scan"]]
    return s["fov"][0] / c["n"], s["fov"][2] / c["nz"], s["det"][0] / c["nu"], s["det"][1] / c["nv"]


def _geometry(c):
    kind = {"fan": "fan2d", "saddle": "noncirc3d"}.get(c["scan"], "circ3d")
    dx, dz, du, dv = _steps(c)
    return ct.Geometry(kind, "curved" if c["scan"] == "curved" else "flat", c["n"], c["n"], c["nz"], dx, dx, dz,
                       c["nu"], c["nv"], du, dv, c["views"], **_params(c))


def _frames(c):
    """Source, detector centre, e_u, e_v and normal of every view (64-bit arrays, nview x 3)."""
    p, nv = _params(c), c["views"]
    get = lambda k: np.broadcast_to(np.asarray(p.get(k, 0.0), dtype=np.float64), (nv,))  # noqa: E731
    th, ph, ps = get("theta"), get("phi"), get("psi")
    zero, one = np.zeros(nv), np.ones(nv)

    def mat(rows):
        return np.stack([np.stack(r, -1) for r in rows], -2)
    Rz = mat([[np.cos(th), -np.sin(th), zero], [np.sin(th), np.cos(th), zero], [zero, zero, one]])
    Rx = mat([[one, zero, zero], [zero, np.cos(ph), -np.sin(ph)], [zero, np.sin(ph), np.cos(ph)]])
    Ry = mat([[np.cos(ps), zero, np.sin(ps)], [zero, one, zero], [-np.sin(ps), zero, np.cos(ps)]])
    R = Rz @ Rx @ Ry
    turn = lambda a: np.einsum("vij,vj->vi", R, np.stack(a, -1))  # noqa: E731
    sad, sdd = get("sad"), get("sdd")
    src = turn([get("x_src"), sad, get("z_src")])
    cen = turn([-get("u_ofst"), sad - sdd, -get("v_ofst")])
    eu, ev = turn([one, zero, zero]), turn([zero, zero, one])
    return src, cen, eu, ev, np.cross(eu, ev)


# ------------------------------------------------------------ inputs
def _bodies(c, seed):
    """Ellipsoids (centre, semi-axes, angle about z, value per mm) inside the field of view."""
    rng = np.random.default_rng(seed)
    half = np.array(SCANS[c["scan"]]["fov"]) / 2
    for _ in range(BODIES):
        cen = rng.uniform(-0.45, 0.45, 3) * half
        axes = rng.uniform(0.08, 0.5, 3) * half
        if c["scan"] == "fan":
            cen[2], axes[2] = 0.0, 1e6
        yield cen, axes, rng.uniform(0, math.pi), rng.uniform(0.002, 0.012)


def _volume(c, seed):
    """A voxelised phantom, batch x [nz x] n x n, 32 bits."""
    dx, dz, _, _ = _steps(c)
    ax = lambda m, h: (torch.arange(m, device="cuda", dtype=torch.float32) - (m - 1) / 2) * h  # noqa: E731
    X, Y, Z = ax(c["n"], dx).view(1, 1, -1), ax(c["n"], dx).view(1, -1, 1), ax(c["nz"], dz).view(-1, 1, 1)
    out = torch.zeros(c["batch"], c["nz"], c["n"], c["n"], device="cuda")
    for b in range(c["batch"]):
        for cen, axes, t, val in _bodies(c, seed * 16 + b):
            p = ((X - cen[0]) * math.cos(t) + (Y - cen[1]) * math.sin(t)) / axes[0]
            q = ((Y - cen[1]) * math.cos(t) - (X - cen[0]) * math.sin(t)) / axes[1]
            out[b] += val * ((p * p + q * q + ((Z - cen[2]) / axes[2]) ** 2) <= 1)
    return out


def _measured(c, seed):
    """Line integrals of a phantom along every cell's central ray with 0.5 % noise, batch x views x nv x nu, 32 bits."""
    _, _, du, dv = _steps(c)
    src, cen, eu, ev, nn = (torch.as_tensor(a, device="cuda", dtype=torch.float32) for a in _frames(c))
    u = (torch.arange(c["nu"], device="cuda") - (c["nu"] - 1) / 2) * du
    v = (torch.arange(c["nv"], device="cuda") - (c["nv"] - 1) / 2) * dv
    noise = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.zeros(c["batch"], c["views"], c["nv"], c["nu"], device="cuda")
    step = max(1, int(16e6 // (c["nu"] * c["nv"])))
    for v0 in range(0, c["views"], step):
        part = slice(v0, v0 + step)
        at = lambda e, k: e[part, k].view(-1, 1, 1)  # noqa: E731
        D = ((cen - src) * nn).sum(-1)[part].view(-1, 1, 1)
        if c["scan"] == "curved":
            lat, dep = D * torch.sin(u / D), D * torch.cos(u / D)
        else:
            lat, dep = u + ((cen - src) * eu).sum(-1)[part].view(-1, 1, 1), D
        hgt = v.view(1, -1, 1) + ((cen - src) * ev).sum(-1)[part].view(-1, 1, 1)
        d = [lat * at(eu, k) + hgt * at(ev, k) + dep * at(nn, k) for k in range(3)]
        size = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        for b in range(c["batch"]):
            for bc, axes, t, val in _bodies(c, seed * 16 + b + 7):
                ct_, st_ = math.cos(t), math.sin(t)
                w = [at(src, k) - float(bc[k]) for k in range(3)]
                W = [(w[0] * ct_ + w[1] * st_) / axes[0], (w[1] * ct_ - w[0] * st_) / axes[1], w[2] / axes[2]]
                E = [(d[0] * ct_ + d[1] * st_) / axes[0], (d[1] * ct_ - d[0] * st_) / axes[1], d[2] / axes[2]]
                A = E[0] ** 2 + E[1] ** 2 + E[2] ** 2
                B = E[0] * W[0] + E[1] * W[1] + E[2] * W[2]
                C = W[0] ** 2 + W[1] ** 2 + W[2] ** 2 - 1
                out[b, part] += val * size * 2 * torch.sqrt(torch.clamp(B * B - A * C, min=0)) / A
    return out * (1 + 0.005 * torch.randn(out.shape, device="cuda", generator=noise))


def _inputs(c, seed):
    T = DTYPES[c["dtype"]]
    lead = () if c["batch"] == 1 else (c["batch"],)
    flat = c["scan"] == "fan"
    y = _measured(c, seed).to(T)
    y = y.reshape(lead + ((c["views"], c["nu"]) if flat else (c["views"], c["nv"], c["nu"])))
    x = None
    if c["op"] in ("pair", "grad"):
        x = _volume(c, seed).to(T)
        x = x.reshape(lead + ((c["n"], c["n"]) if flat else (c["nz"], c["n"], c["n"])))
    return x, y


def _rate(c):
    """A gradient step below 1 / ||A||^2: the product of the largest row and column sums, bounded."""
    s, (dx, dz, du, dv) = SCANS[c["scan"]], _steps(c)
    near = s["sdd"] / (s["sad"] - s["fov"][0] / math.sqrt(2))
    col = c["views"] * 1.5 * dx * near * dx / du * (1.0 if c["scan"] == "fan" else near * dz / dv)
    return 1.0 / (1.6 * s["fov"][0] * col)


def prepare(case, seed):
    x, y = _inputs(case, seed)
    s = dict(case=case, geom=_geometry(case), x=x, y=y)
    if case["op"] == "grad":
        s["A"] = ct.Projector(s["geom"], "proj", case["projector"], "forward")
        s["x"].requires_grad_(True)
    if case["op"] == "mbir":
        s["lr"] = _rate(case)
    return s


def run(s):
    c, g = s["case"], s["geom"]
    if c["op"] == "pair":
        return {"sino": ct.forward(g, s["x"], c["projector"]), "vol": ct.back(g, s["y"], c["adjoint"])}
    if c["op"] == "grad":
        s["x"].grad = None
        r = s["A"](s["x"]) - s["y"]
        loss = 0.5 * (r * r).sum()
        loss.backward()
        return {"residual": r.detach(), "grad": s["x"].grad}
    if c["op"] == "mbir":
        return {"vol": mbir.ls_gradient_descent(g, s["y"], c["projector"], c["steps"], lr=s["lr"])}
    if c["projector"] == "voxel":
        return {"vol": ct.fbp(g, s["y"])}
    q = ct.ramp_filter(g, s["y"])
    return {"filtered": q, "vol": ct.back(g, q, c["projector"], mode="recon")}


def work(case):
    c = case
    vox = c["batch"] * c["n"] * c["n"] * c["nz"]
    cells = c["batch"] * c["views"] * c["nu"] * c["nv"]
    size = 4 if c["dtype"] == "f32" else 2
    # each pass reads one side and writes the other; a filter writes and reads its rows once more
    io = _passes(c) * (vox + cells) + (2 * cells if c["op"] == "fbp" else 0)
    # operations of one (voxel, view) pair: footprint weights applied and summed
    per = {"sf": 30, "dd": 24, "voxel": 16, "ray": 30, "sftt": 60}[c["projector"]] * (3 if c["scan"] == "saddle" else 1)
    return {"bytes": float(size * io), "flops": float(per * _updates(c))}


# ------------------------------------------------------------ the projectors in 64 bits
#: (voxel, view) pairs whose 64-bit restatement stays below 20 seconds
EXACT_MOST = {"fan": 6e9, "circ": 14e9, "curved": 14e9, "saddle": 4e9}


def _ramp_at(x, e):
    """Integral up to x of the ramp rising from 0 at 0 to 1 at e and staying there."""
    t = torch.minimum(x.clamp(min=0), e)
    return t * t * 0.5 / e.clamp(min=1e-200) + (x - e).clamp(min=0)


def _trapezoid(k, f):
    """Integral up to f of the unit trapezoid with sorted knots k[0..3]."""
    return _ramp_at(f - k[0], k[1] - k[0]) - _ramp_at(f - k[2], k[3] - k[2])


def _sorted(t):
    return torch.sort(torch.stack(torch.broadcast_tensors(*t)), 0).values


class _View:
    """One view's mapping and weights, for all voxels: arrays of (nz, ncol) or (1, ncol)."""

    def __init__(self, c, frames, v, X, Y, Z, beta):
        self.c, self.flat2d = c, c["scan"] == "fan"
        self.dx, self.dz, self.du, self.dv = _steps(c)
        src, cen, eu, ev, nn = (a[v] for a in frames)
        self.src, self.cen, self.eu, self.ev, self.nn, self.beta = src, cen, eu, ev, nn, beta
        self.D = float(np.dot(cen - src, nn))
        self.u0, self.v0 = float(np.dot(cen - src, eu)), float(np.dot(cen - src, ev))
        self.main_y = abs(cen[1] - src[1]) >= abs(cen[0] - src[0])
        self.wx, self.wy, self.wz = X - src[0], Y - src[1], Z - src[2]
        self.tilted = c["scan"] == "saddle"
        self.curved = c["scan"] == "curved"

    def dots(self, ox=0.0, oy=0.0, oz=0.0, z=True):
        """(w.e_u, w.e_v, w.n) of the voxels' points at an offset; without z, (1, ncol) where the scan is circular."""
        wx, wy = self.wx + ox, self.wy + oy
        wz = self.wz + oz if (z or self.tilted) else 0.0
        f = lambda e: wx * e[0] + wy * e[1] + (wz * e[2] if e[2] != 0 else 0.0)  # noqa: E731
        return f(self.eu), f(self.ev), f(self.nn)

    def fu(self, **at):
        a, _, b = self.dots(z=False, **at)
        u = self.D * (torch.atan2(a, b) if self.curved else a / b) - self.u0
        return u / self.du + (self.c["nu"] - 1) / 2

    def depth(self, **at):
        a, _, b = self.dots(z=False, **at)
        return torch.sqrt(a * a + b * b) if self.curved else b

    def fv(self, **at):
        return (self.D * self.dots(**at)[1] / self.depth(**at) - self.v0) / self.dv + (self.c["nv"] - 1) / 2

    def knots_u(self, projector):
        h = self.dx / 2
        if projector == "dd":
            t = _sorted([self.fu(ox=s * h) if self.main_y else self.fu(oy=s * h) for s in (-1, 1)])
            return torch.stack([t[0], t[0], t[1], t[1]])
        return _sorted([self.fu(ox=p * h, oy=q * h) for p in (-1, 1) for q in (-1, 1)])

    def knots_v(self, projector):
        h = self.dz / 2
        if projector == "sftt":
            hx = self.dx / 2
            n, tiny = self.nn, 1e-7
            near = [(h2 if m < -tiny else -h2) for m, h2 in ((n[0], hx), (n[1], hx))]
            far = [(h2 if m > tiny else -h2) for m, h2 in ((n[0], hx), (n[1], hx))]
            return _sorted([self.fv(ox=o[0], oy=o[1], oz=s) for o in (near, far) for s in (-h, h)])
        t = _sorted([self.fv(oz=s) for s in (-h, h)])
        return torch.stack([t[0], t[0], t[1], t[1]])

    def taps(self, projector, recon):
        """(first cell, [weights]), (first row, [weights]), amplitude per voxel, factor per cell (or None)."""
        if projector == "voxel":
            fu, fv = self.fu(), None if self.flat2d else self.fv()
            u = (torch.floor(fu), [1 - (fu - torch.floor(fu)), fu - torch.floor(fu)])
            v = None if self.flat2d else (torch.floor(fv), [1 - (fv - torch.floor(fv)), fv - torch.floor(fv)])
            area = 1.0
        else:
            k = self.knots_u(projector)
            u, area = self.cells(k), 0.5 * (k[3] - k[0] + k[2] - k[1])
            v = None
            if not self.flat2d:
                k = self.knots_v(projector)
                v = self.cells(k)
                area = area * 0.5 * (k[3] - k[0] + k[2] - k[1])
        dep = self.depth()
        if recon:
            R = -float(np.dot(self.src, self.nn))
            return u, v, self.beta * (1.0 if self.curved else R * self.D) / (dep * dep * area), None
        r = torch.sqrt(self.wx ** 2 + self.wy ** 2 + (0.0 if self.flat2d else self.wz ** 2))
        if projector == "voxel":
            if self.flat2d:
                return u, v, self.dx ** 2 / self.du * r * self.D / dep ** 2, None
            return u, v, self.dx ** 2 * self.dz / (self.du * self.dv) * r * self.D ** 2 / dep ** 3, None
        if projector == "sf":
            return u, v, self.dx * r / torch.maximum(self.wx.abs(), self.wy.abs()), None
        d = self.rays()
        size = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        if projector == "sftt":
            return u, v, 1.0, self.dx * size / torch.maximum(d[0].abs(), d[1].abs())
        return u, v, 1.0, self.dx * size / (d[1] if self.main_y else d[0]).abs()

    def cells(self, k):
        """First cell under the trapezoid k, and the integral over each cell from there on."""
        first = torch.floor(k[0] + 0.5)
        count = int((torch.floor(k[3] + 0.5) - first).max()) + 1
        g = [_trapezoid(k, first + q - 0.5) for q in range(count + 1)]
        return first, [g[q + 1] - g[q] for q in range(count)]

    def rays(self):
        """World vectors from the source to the cell centres, three (nv, nu) arrays."""
        c = self.c
        f = lambda m, h: ((torch.arange(m, device="cuda", dtype=torch.float64) - (m - 1) / 2) * h)  # noqa: E731
        u = f(c["nu"], self.du).view(1, -1) + self.u0
        v = f(c["nv"], self.dv).view(-1, 1) + self.v0
        lat, dep = (self.D * torch.sin(u / self.D), self.D * torch.cos(u / self.D)) if self.curved else (u, self.D)
        if self.flat2d:
            v = torch.zeros_like(v)
        return [lat * self.eu[k] + v * self.ev[k] + dep * self.nn[k] for k in range(3)]

    def segments(self):
        """Siddon: voxel index and length of every piece of every cell's central ray, (cells, pieces)."""
        c = self.c
        d = [t.expand(c["nv"], c["nu"]).reshape(-1, 1) for t in self.rays()]
        n, h = (c["n"], c["n"], c["nz"]), (self.dx, self.dx, self.dz)
        axes = (0, 1) if self.flat2d else (0, 1, 2)
        tin, tout = torch.zeros_like(d[0]), torch.ones_like(d[0])
        planes = []
        for m in axes:
            p = (torch.arange(n[m] + 1, device="cuda", dtype=torch.float64) - n[m] / 2) * h[m] - self.src[m]
            t = p.view(1, -1) / torch.where(d[m] == 0, torch.full_like(d[m], 1e-300), d[m])
            planes.append(t)
            tin = torch.maximum(tin, torch.minimum(t[:, :1], t[:, -1:]))
            tout = torch.minimum(tout, torch.maximum(t[:, :1], t[:, -1:]))
        tout = torch.maximum(tin, tout)
        t = torch.sort(torch.maximum(torch.minimum(torch.cat(planes, 1), tout), tin), 1).values
        size = torch.sqrt(sum(d[m] ** 2 for m in axes))
        w = (t[:, 1:] - t[:, :-1]) * size
        mid = 0.5 * (t[:, 1:] + t[:, :-1])
        i = [torch.floor((self.src[m] + mid * d[m]) / h[m] + n[m] / 2).clamp(0, n[m] - 1).long() for m in axes]
        k = i[2] if len(axes) == 3 else 0
        return (k * n[1] + i[1]) * n[0] + i[0], w


def _weights(tap, size):
    """[(index, weight)] of a tap list, off-detector cells at weight zero."""
    first, ws = tap
    out = []
    for q, w in enumerate(ws):
        at = first + q
        ok = (at >= 0) & (at < size)
        out.append((at.clamp(0, size - 1).long(), torch.where(ok, w, torch.zeros((), device="cuda", dtype=w.dtype))))
    return out


class _Exact:
    def __init__(self, c):
        self.c, self.frames = c, _frames(c)
        dx, dz, _, _ = _steps(c)
        f = lambda m, h: (torch.arange(m, device="cuda", dtype=torch.float64) - (m - 1) / 2) * h  # noqa: E731
        n = c["n"]
        self.X, self.Y = f(n, dx).repeat(n).view(1, -1), f(n, dx).repeat_interleave(n).view(1, -1)
        self.Z = f(c["nz"], dz if c["scan"] != "fan" else 0.0).view(-1, 1)

    def views(self):
        for v in range(self.c["views"]):
            yield v, _View(self.c, self.frames, v, self.X, self.Y, self.Z, 2 * math.pi / self.c["views"])

    def forward(self, x, projector):
        """x: (batch, nz, ncol) -> (batch, views, nv, nu)."""
        c = self.c
        nv, nu, nb = c["nv"], c["nu"], c["batch"]
        out = torch.zeros(nb, c["views"], nv, nu, device="cuda", dtype=torch.float64)
        for v, view in self.views():
            if projector == "ray":
                at, w = view.segments()
                for b in range(nb):
                    out[b, v] = (w * x[b].reshape(-1)[at]).sum(1).view(nv, nu)
                continue
            tu, tv, amp, factor = view.taps(projector, False)
            us = _weights(tu, nu)
            vs = [(0, 1.0)] if tv is None else _weights(tv, nv)
            for b in range(nb):
                val = x[b] * amp
                if view.tilted:
                    y = torch.zeros(nv * nu, device="cuda", dtype=torch.float64)
                    for rb, wv in vs:
                        t = val * wv
                        for ca, wu in us:
                            y.index_add_(0, (rb * nu + ca).view(-1), (t * wu).view(-1))
                    y = y.view(nv, nu)
                else:  # down each column first, then across
                    ncol = x.shape[2]
                    if tv is None:
                        Z = val
                    else:
                        Z = torch.zeros(nv * ncol, device="cuda", dtype=torch.float64)
                        col = torch.arange(ncol, device="cuda").view(1, -1)
                        for rb, wv in vs:
                            Z.index_add_(0, (rb * ncol + col).view(-1), (val * wv).view(-1))
                    Z = Z.view(-1, ncol).t().contiguous()
                    y = torch.zeros(nu, nv, device="cuda", dtype=torch.float64)
                    for ca, wu in us:
                        y.index_add_(0, ca.view(-1), Z * wu.view(-1, 1))
                    y = y.t()
                out[b, v] = y if factor is None else y * factor
        return out

    def back(self, y, projector, recon=False):
        """y: (batch, views, nv, nu) -> (batch, nz, ncol)."""
        c = self.c
        nv, nu, nb = c["nv"], c["nu"], c["batch"]
        out = torch.zeros(nb, c["nz"], c["n"] ** 2, device="cuda", dtype=torch.float64)
        for v, view in self.views():
            if projector == "ray":
                at, w = view.segments()
                for b in range(nb):
                    out[b].view(-1).index_add_(0, at.view(-1), (w * y[b, v].reshape(-1, 1)).view(-1))
                continue
            tu, tv, amp, factor = view.taps(projector, recon)
            us = _weights(tu, nu)
            vs = [(0, 1.0)] if tv is None else _weights(tv, nv)
            for b in range(nb):
                s = y[b, v] if factor is None else y[b, v] * factor
                if view.tilted:
                    flat, acc = s.reshape(-1), 0.0
                    for rb, wv in vs:
                        row = 0.0
                        for ca, wu in us:
                            row = row + wu * flat[rb * nu + ca]
                        acc = acc + wv * row
                else:
                    R = 0.0
                    for ca, wu in us:
                        R = R + wu.view(1, -1) * s[:, ca.view(-1)]
                    acc = R if tv is None else sum(wv * R.gather(0, rb) for rb, wv in vs)
                out[b] += amp * acc
        return out

    def filter(self, y):
        """The pre-weighted ramp filter of every row."""
        c = self.c
        _, _, du, dv = _steps(c)
        nu = c["nu"]
        f = lambda m: torch.arange(m, device="cuda", dtype=torch.float64) - (m - 1) / 2  # noqa: E731
        out = torch.empty_like(y)
        for v, view in self.views():
            D, R = view.D, -float(np.dot(view.src, view.nn))
            up = (f(nu) * du + view.u0).view(1, -1)
            vp = torch.zeros(1, 1, device="cuda", dtype=torch.float64) if view.flat2d else (f(c["nv"]) * dv + view.v0).view(-1, 1)
            if view.curved:
                wgt, step = R * torch.cos(up / D) * D / torch.sqrt(D * D + vp * vp), du / D
            else:
                wgt, step = D / torch.sqrt(D * D + up * up + vp * vp), du
            k = torch.arange(nu, device="cuda").view(1, -1) - torch.arange(nu, device="cuda").view(-1, 1)
            den = torch.sin(k * step) if view.curved else k * step
            h = torch.where(k % 2 == 0, torch.zeros((), device="cuda", dtype=torch.float64),
                            -1 / (2 * math.pi ** 2 * torch.where(k == 0, torch.ones_like(den), den) ** 2))
            h = h + torch.eye(nu, device="cuda", dtype=torch.float64) / (8 * step ** 2)
            out[:, v] = step * (y[:, v] * wgt) @ h
        return out


def exact(case, seed):
    c = case
    if _updates(c) * (3 if c["projector"] == "ray" else 1) > EXACT_MOST[c["scan"]]:
        return None
    x, y = _inputs(c, seed)
    E = _Exact(c)
    shape_x = () if c["batch"] == 1 else (c["batch"],)
    shape_y = shape_x + ((c["views"], c["nu"]) if c["scan"] == "fan" else (c["views"], c["nv"], c["nu"]))
    shape_x = shape_x + ((c["n"], c["n"]) if c["scan"] == "fan" else (c["nz"], c["n"], c["n"]))
    y = y.double().view(c["batch"], c["views"], c["nv"], c["nu"])
    x = None if x is None else x.double().view(c["batch"], c["nz"], -1)
    if c["op"] == "pair":
        return {"sino": E.forward(x, c["projector"]).view(shape_y), "vol": E.back(y, c["adjoint"]).view(shape_x)}
    if c["op"] == "grad":
        r = E.forward(x, c["projector"]) - y
        return {"residual": r.view(shape_y), "grad": E.back(r, c["projector"]).view(shape_x)}
    if c["op"] == "mbir":
        x = torch.zeros(c["batch"], c["nz"], c["n"] ** 2, device="cuda", dtype=torch.float64)
        for k in range(c["steps"]):
            r = E.forward(x, c["projector"]) - y if k else -y
            x = x - _rate(c) * E.back(r, c["projector"])
        return {"vol": x.view(shape_x)}
    q = E.filter(y)
    vol = E.back(q, c["projector"], recon=True).view(shape_x)
    return {"vol": vol} if c["projector"] == "voxel" else {"filtered": q.view(shape_y), "vol": vol}
