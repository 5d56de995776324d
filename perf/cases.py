"""The work that a user of this framework has it do, as measurable cases.

Every case goes through a public entry point (``forward``, ``adjoint``,
``autograd.project``, ``recon.cgls``, ``Batch.forward``) on a cone-beam scan
like those of the benchmark and the tests:

* ``op``      -- which entry point; "step" is one gradient step (projection,
                 squared-error loss, backward), "cgls" a short reconstruction,
                 "batch" many few-view problems in one call;
* ``nx, ny, nz``, ``hx, hy, hz`` -- volume grid and voxel size;
* ``nu, nv, views``  -- detector columns and rows, views;
* ``half_angle``     -- cone half-angle (degrees) on the inscribed cylinder;
* ``dtype``, ``weight`` -- volume storage, interpolation weight;
* ``fov``     -- whether rays are clipped to the field-of-view cylinder;
* ``start``   -- angle of the first view (degrees);
* ``arc``     -- degrees covered by the views (equidistant, end excluded);
* ``pitch``   -- helical travel along z per turn, as a part of the height;
* ``shift_u, shift_v`` -- detector offset in pixels;
* ``tilt``    -- calibrated misalignment (degrees) of the detector's axes:
                 0 is the aligned scanner, whose detector rows run along z.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1609_00958_gb300 as gjp
from paper_1609_00958_gb300 import autograd, recon

TYPES = {"float32": torch.float32, "bfloat16": torch.bfloat16, "float16": torch.float16}
DEV = "cuda"
# exact() stays below about 20 seconds up to this many (ray, plane) samples
EXACT_SAMPLES = 8.0e10


def _case(name, op, n, det, views, **more):
    c = {"name": name, "op": op, "nx": n[0], "ny": n[1], "nz": n[2], "hx": 1.0, "hy": 1.0, "hz": 1.0,
         "nu": det[0], "nv": det[1], "views": views, "half_angle": 10.0, "dtype": "float32", "weight": "lin",
         "fov": False, "start": 0.0, "arc": 360.0, "pitch": 0.0, "shift_u": 0.0, "shift_v": 0.0, "tilt": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # One digitally rendered radiograph, as 2D/3D registration asks for by the hundred: a call's latency.
        _case("radiograph_256", "forward", (256, 256, 256), (256, 256), 1, start=30.0),
        # The small scan of the benchmark, projected and backprojected: launches and per-ray setup count.
        _case("forward_64", "forward", (64, 64, 64), (64, 64), 32, half_angle=7.0),
        _case("adjoint_64", "adjoint", (64, 64, 64), (64, 64), 32, half_angle=7.0),
        # The benchmark's full scan: 512^3, 360 views, in both storage types it reports, and its backprojection.
        _case("forward_512", "forward", (512, 512, 512), (512, 512), 360),
        _case("forward_512_bf16", "forward", (512, 512, 512), (512, 512), 360, dtype="bfloat16"),
        _case("adjoint_512", "adjoint", (512, 512, 512), (512, 512), 360),
        # The precision form's grid in half storage, an ordered subset of its views as iterative solvers use them.
        _case("forward_1024_f16", "forward", (1024, 1024, 1024), (1024, 1024), 60, dtype="float16"),
        # A scan of a user's own: odd sizes, anisotropic voxels, an offset detector on a helix, smooth weights,
        # rays clipped to the scanner's field of view.
        _case("forward_odd_helix", "forward", (331, 287, 203), (301, 243), 123, hx=0.8, hy=0.9, hz=1.25,
              dtype="float16", weight="spl", fov=True, start=3.7, pitch=0.3, shift_u=2.25, shift_v=-3.5),
        _case("adjoint_odd", "adjoint", (309, 333, 179), (287, 211), 97, hx=0.9, hy=1.0, hz=1.3, weight="spl",
              start=1.3, shift_u=-1.75, shift_v=2.5),
        # A gradient step on a scanner whose calibration found its detector slightly tilted.
        _case("step_tilted_192", "step", (192, 192, 192), (192, 192), 96, tilt=0.7, start=0.5),
        # Two iterations of the differentiation form's reconstruction.
        _case("cgls_256", "cgls", (256, 256, 256), (256, 256), 180, start=0.25),
        # The benchmark's mix of few-view problems (tomosynthesis-like), in one batch.
        _case("batch_few_views", "batch", (192, 192, 192), (192, 192), 16),
    ]


def draw(rng):
    op = rng.choice(["forward", "forward", "adjoint", "adjoint", "step", "cgls", "batch"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    edge = log(40, 600)
    n = tuple(max(24, int(edge * rng.uniform(0.7, 1.15))) for _ in range(3))
    if rng.random() < 0.35:
        n = (edge,) * 3
    if rng.random() < 0.15:
        n = (n[0], n[1], max(24, n[2] // 4))
    det = (max(24, int(max(n[0], n[1]) * rng.uniform(0.75, 1.2))), max(24, int(n[2] * rng.uniform(0.75, 1.2))))
    views = log(1, 400)
    limit = {"forward": 2.4e10, "adjoint": 1.6e10, "step": 5.0e9, "cgls": 3.0e9, "batch": 1.0}[op]
    views = max(1, min(views, int(limit / (det[0] * det[1] * max(n)))))
    aligned = rng.random() < 0.85
    c = _case("", op, n, det, views, half_angle=rng.uniform(4.0, 14.0), start=rng.uniform(0.0, 44.0),
              arc=rng.choice([360.0, 360.0, 200.0]), shift_u=rng.uniform(-4.0, 4.0), shift_v=rng.uniform(-4.0, 4.0))
    if rng.random() < 0.4:
        c.update(hx=rng.uniform(0.7, 1.4), hy=rng.uniform(0.7, 1.4), hz=rng.uniform(0.6, 1.6))
    if rng.random() < 0.2:
        c["weight"] = "spl"
    if rng.random() < 0.2:
        c["pitch"] = rng.uniform(0.05, 0.5)
    if op == "forward":
        c["dtype"] = rng.choice(["float32", "float32", "bfloat16", "float16"])
        c["fov"] = rng.random() < 0.15
    if op == "batch":
        c.update(_case("", op, (rng.choice([96, 128, 160, 192]),) * 3, (rng.randint(96, 192),) * 2, rng.randint(6, 16),
                       start=rng.uniform(0.0, 44.0)))
    elif not aligned:
        c["tilt"] = rng.uniform(0.1, 2.0)
        c["fov"] = False
    del c["name"]
    return c


# --- the scan ---------------------------------------------------------------


class _Scan:
    """The case's geometry as float64 host arrays, as a scanner's calibration gives it."""

    def __init__(self, c):
        self.n = (c["nx"], c["ny"], c["nz"])
        self.h = (c["hx"], c["hy"], c["hz"])
        self.nu, self.nv, self.views = c["nu"], c["nv"], c["views"]
        a = math.radians(c["half_angle"])
        width = max(self.n[0] * self.h[0], self.n[1] * self.h[1])
        height = self.n[2] * self.h[2]
        self.width = width
        d_so = 0.5 * width / math.sin(a)
        d_sd = 2.0 * d_so
        pu = 2.0 * d_sd * math.tan(a) / self.nu
        pv = 2.0 * d_sd * math.tan(a) * (height / width) / self.nv
        k = np.arange(self.views)
        th = np.radians(c["start"] + c["arc"] * k / self.views)
        co, si, ze = np.cos(th), np.sin(th), np.zeros(self.views)
        z = c["pitch"] * height * (c["arc"] / 360.0) * ((k + 0.5) / self.views - 0.5)
        eu = np.stack([-si, co, ze], 1)
        ev = np.stack([ze, ze, ze + 1.0], 1)
        if c["tilt"]:
            t = math.radians(c["tilt"])
            nrm = np.stack([co, si, ze], 1)
            # in-plane rotation, then a lean of the rows towards the source
            eu, ev = math.cos(t) * eu + math.sin(t) * ev, -math.sin(t) * eu + math.cos(t) * ev
            ev = math.cos(0.5 * t) * ev + math.sin(0.5 * t) * nrm
        centre = np.stack([-(d_sd - d_so) * co, -(d_sd - d_so) * si, z], 1)
        self.src = np.stack([d_so * co, d_so * si, z], 1)
        self.du, self.dv = eu * pu, ev * pv
        self.org = (centre + (c["shift_u"] - 0.5 * (self.nu - 1)) * self.du
                    + (c["shift_v"] - 0.5 * (self.nv - 1)) * self.dv)
        self.fov = 0.47 * width if c["fov"] else 0.0

    def handle(self, weight):
        g = gjp.Geometry(self.src, self.org, self.du, self.dv, self.nu, self.nv, weight=weight)
        if self.fov:
            g.set_fov(self.fov)
        return g


def _problems(c):
    """The problems of a "batch" case: few-view scans of mixed sizes and storage types, the case's own the largest."""
    rng = np.random.default_rng(c["nx"] * 1009 + c["nu"] * 31 + c["views"])
    out = []
    for k in range(24):
        p = dict(c, op="forward")
        if k:
            e = max(48, int(c["nx"] * rng.choice([0.5, 0.667, 0.833, 1.0])))
            d = int(rng.integers(c["nu"] // 2, c["nu"] + 1))
            p.update(nx=e, ny=e, nz=e, nu=d, nv=d, views=int(rng.integers(2, c["views"] + 1)),
                     half_angle=float(rng.uniform(5.0, 15.0)))
        p["dtype"] = ["float32", "bfloat16"][int(rng.integers(0, 2))]
        out.append(p)
    return out


def _volume(s, gen):
    """An ellipsoidal body with a denser shell and a textured interior, attenuation values in [0, 1.3); zero outside."""
    ax = [torch.linspace(-1.0, 1.0, k, device=DEV) for k in s.n]
    r2 = (ax[0] / 0.86).square()[:, None, None] + (ax[1] / 0.9).square()[None, :, None]
    r2 = r2 + (ax[2] / 0.97).square()[None, None, :]
    v = torch.rand(s.n, generator=gen, device=DEV)
    v.mul_(0.3).add_(0.3).add_((r2 > 0.85).to(v.dtype), alpha=0.7)
    if s.fov:
        # nothing lies near the wall of the field of view
        x = (torch.arange(s.n[0], device=DEV) - 0.5 * (s.n[0] - 1)) * s.h[0]
        y = (torch.arange(s.n[1], device=DEV) - 0.5 * (s.n[1] - 1)) * s.h[1]
        keep = x.square()[:, None] + y.square()[None, :] < (s.fov - 3.0 * max(s.h[0], s.h[1])) ** 2
        v.mul_(keep[:, :, None])
    return v.mul_(r2 <= 1.0)


def _rows(s, gen):
    """Projection-like values: a smooth profile with noise, signed as residuals and filtered projections are."""
    u = torch.linspace(-1.0, 1.0, s.nu, device=DEV)
    v = torch.linspace(-1.0, 1.0, s.nv, device=DEV)
    y = torch.randn((s.views, s.nv, s.nu), generator=gen, device=DEV)
    return y.mul_(0.3).add_(1.0 - 0.7 * (v.square()[:, None] + u.square()[None, :]))


# --- the three functions that are timed ----------------------------------------


def _inputs(c, seed):
    """The case's tensors, from the seed alone."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    if c["op"] == "batch":
        return {"vols": [_volume(_Scan(p), gen).to(TYPES[p["dtype"]]) for p in _problems(c)]}
    s, st = _Scan(c), {}
    if c["op"] in ("forward", "step"):
        st["vol"] = _volume(s, gen).to(TYPES[c["dtype"]])
    if c["op"] in ("adjoint", "step", "cgls"):
        st["rows"] = _rows(s, gen)
    if c["op"] in ("step", "cgls"):
        st["rows"].mul_(0.2 * s.width)
    return st


def prepare(case, seed):
    c = case
    st = _inputs(c, seed)
    st["op"] = c["op"]
    if c["op"] == "batch":
        recs = []
        for p, vol in zip(_problems(c), st["vols"]):
            s = _Scan(p)
            g = s.handle(p["weight"])
            recs.append((vol, g, s.h, None, torch.empty(g.proj_shape, dtype=torch.float32, device=DEV)))
        st["batch"] = gjp.Batch(recs)
        return st
    st["scan"] = _Scan(c)
    st["geom"] = st["scan"].handle(c["weight"])
    if c["op"] == "step":
        st["vol"].requires_grad_(True)
    return st


def run(state):
    op = state["op"]
    if op == "batch":
        return state["batch"].forward()
    s, g = state["scan"], state["geom"]
    if op == "forward":
        return gjp.forward(state["vol"], g, s.h)
    if op == "adjoint":
        return gjp.adjoint(state["rows"], g, s.n, s.h)
    if op == "step":
        proj = autograd.project(state["vol"], g, s.h)
        loss = 0.5 * (proj - state["rows"]).square().mean()
        (grad,) = torch.autograd.grad(loss, state["vol"])
        return {"proj": proj.detach(), "grad": grad}
    x, history = recon.cgls(state["rows"], g, s.n, 2, s.h)
    return {"x": x, "residual": history.residual}


def _samples(c):
    """(ray, plane) samples of the case's scan, from a grid of rays over a few views."""
    s = _Scan(c)
    n = np.array(s.n, float)
    total = 0.0
    ks = np.unique(np.linspace(0, s.views - 1, min(s.views, 12)).astype(int))
    iu = np.linspace(0, s.nu - 1, min(s.nu, 24))
    iv = np.linspace(0, s.nv - 1, min(s.nv, 24))
    for k in ks:
        src = s.src[k] / s.h + 0.5 * (n - 1)
        d = (s.org[k] + iu[:, None, None] * s.du[k] + iv[None, :, None] * s.dv[k]) / s.h + 0.5 * (n - 1)
        r = (d - src).reshape(-1, 3)
        m = np.argmax(np.abs(r), 1)
        rm = np.take_along_axis(r, m[:, None], 1)[:, 0]
        t0, t1 = (0 - src[m]) / rm, (n[m] - 1 - src[m]) / rm
        lo, hi = np.minimum(t0, t1), np.maximum(t0, t1)
        for a in range(3):
            with np.errstate(divide="ignore", invalid="ignore"):
                e0, e1 = (-1 - src[a]) / r[:, a], (n[a] - src[a]) / r[:, a]
            other = m != a
            lo = np.where(other, np.fmax(lo, np.fmin(e0, e1)), lo)
            hi = np.where(other, np.fmin(hi, np.fmax(e0, e1)), hi)
        total += np.maximum(0.0, (hi - lo) * np.abs(rm)).mean()
    return total / len(ks) * s.views * s.nu * s.nv


def work(case):
    """Bytes: volume and projections, each once per pass over them.  Operations of one sample (Eq. 12, accumulation):
    three interpolations of 3, one addition, two position updates."""
    if case["op"] == "batch":
        ws = [work(p) for p in _problems(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    c = case
    size = 4 if c["dtype"] == "float32" else 2
    vol, proj = c["nx"] * c["ny"] * c["nz"] * size, c["nu"] * c["nv"] * c["views"] * 4
    one = 12.0 * _samples(c)
    if c["op"] in ("forward", "adjoint"):
        return {"bytes": vol + proj, "flops": one}
    if c["op"] == "step":
        return {"bytes": 2 * vol + 2 * proj, "flops": 2 * one}
    # two iterations: A^T b first, then A p and A^T r each time
    return {"bytes": vol + proj, "flops": 5 * one}


# --- 64-bit values ----------------------------------------------------------------


def _joseph(s, weight, vol=None, rows=None):
    """The projections of ``vol`` or the backprojection of ``rows``, sample by sample in float64."""
    n, f64 = s.n, torch.float64
    pad = (n[0] + 3, n[1] + 3, n[2] + 3)                   # zero border: one voxel below, two above
    stride = (pad[1] * pad[2], pad[2], 1)
    if vol is not None:
        work_vol = torch.zeros(pad, dtype=f64, device=DEV)
        work_vol[1:-2, 1:-2, 1:-2] = vol
        flat = work_vol.view(-1)
        out = torch.zeros((s.views, s.nv * s.nu), dtype=f64, device=DEV)
    else:
        flat = torch.zeros(pad[0] * pad[1] * pad[2], dtype=f64, device=DEV)
    h = torch.tensor(s.h, dtype=f64, device=DEV)
    off = torch.tensor([0.5 * (k - 1) for k in n], dtype=f64, device=DEV)
    iu = torch.arange(s.nu, dtype=f64, device=DEV)
    iv = torch.arange(s.nv, dtype=f64, device=DEV)

    def arr(x):
        return torch.tensor(x, dtype=f64, device=DEV)

    def upper(d):
        return d if weight == "lin" else d * d * (3.0 - 2.0 * d)

    for k in range(s.views):
        src = arr(s.src[k]) / h + off
        d = arr(s.org[k]) + iv[:, None, None] * arr(s.dv[k]) + iu[None, :, None] * arr(s.du[k])
        r_all = (d / h + off - src).view(-1, 3)
        m_all = r_all.abs().argmax(1)
        for m in range(3):
            sel = torch.nonzero(m_all == m).view(-1)
            if not len(sel):
                continue
            a, b = [q for q in range(3) if q != m]
            r = r_all[sel]
            ga, gb = r[:, a] / r[:, m], r[:, b] / r[:, m]
            step = (h[m] ** 2 + (h[a] * ga) ** 2 + (h[b] * gb) ** 2).sqrt()
            y = rows[k].reshape(-1)[sel].to(f64) * step if rows is not None else None
            acc = torch.zeros(len(sel), dtype=f64, device=DEV)
            chunk = max(1, 40_000_000 // len(sel))
            for i0 in range(0, n[m], chunk):
                i = torch.arange(i0, min(n[m], i0 + chunk), dtype=f64, device=DEV)[:, None]
                pa = src[a] + (i - src[m]) * ga
                pb = src[b] + (i - src[m]) * gb
                keep = None
                if s.fov:
                    q = {m: i, a: pa, b: pb}
                    keep = ((q[0] - off[0]) * h[0]).square() + ((q[1] - off[1]) * h[1]).square() <= s.fov ** 2
                pa.clamp_(-1.0, float(n[a]))
                pb.clamp_(-1.0, float(n[b]))
                fa, fb = pa.floor(), pb.floor()
                idx = ((i + 1) * stride[m] + (fa + 1) * stride[a] + (fb + 1) * stride[b]).to(torch.int64)
                da, db = upper(pa.sub_(fa)), upper(pb.sub_(fb))
                if vol is not None:
                    lo = torch.take(flat, idx)
                    lo += db * (torch.take(flat, idx + stride[b]) - lo)
                    idx += stride[a]
                    hi = torch.take(flat, idx)
                    hi += db * (torch.take(flat, idx + stride[b]) - hi)
                    val = lo + da * (hi - lo)
                    acc += (val * keep if keep is not None else val).sum(0)
                else:
                    yk = y * keep if keep is not None else y.expand_as(da)
                    for w, o in (((1 - da) * (1 - db), 0), ((1 - da) * db, stride[b]), (da * (1 - db), stride[a]),
                                 (da * db, stride[a] + stride[b])):
                        flat.index_add_(0, (idx + o).view(-1), (w * yk).view(-1))
            if vol is not None:
                out[k, sel] = acc * step
    if vol is not None:
        return out.view(s.views, s.nv, s.nu)
    return flat.view(pad)[1:-2, 1:-2, 1:-2].contiguous()


def exact(case, seed):
    c = case
    passes = {"forward": 1, "adjoint": 2, "step": 3, "cgls": 8, "batch": 1}[c["op"]]
    if c["op"] != "batch" and passes * _samples(c) > EXACT_SAMPLES:
        return None
    st = _inputs(c, seed)
    if c["op"] == "batch":
        return [_joseph(_Scan(p), p["weight"], vol=v) for p, v in zip(_problems(c), st["vols"])]
    s, w = _Scan(c), c["weight"]
    if c["op"] == "forward":
        return _joseph(s, w, vol=st["vol"])
    if c["op"] == "adjoint":
        return _joseph(s, w, rows=st["rows"])
    if c["op"] == "step":
        proj = _joseph(s, w, vol=st["vol"])
        return {"proj": proj, "grad": _joseph(s, w, rows=(proj - st["rows"].double()) / proj.numel())}
    # conjugate gradients on the normal equations, from zero
    b = st["rows"].double()
    x = torch.zeros(s.n, dtype=torch.float64, device=DEV)
    r, res = b.clone(), [float(b.norm())]
    grad = _joseph(s, w, rows=r)
    p, gamma = grad.clone(), grad.square().sum()
    for _ in range(2):
        q = _joseph(s, w, vol=p)
        alpha = gamma / q.square().sum()
        x += alpha * p
        r -= alpha * q
        res.append(float(r.norm()))
        grad = _joseph(s, w, rows=r)
        new = grad.square().sum()
        p = grad + (new / gamma) * p
        gamma = new
    return {"x": x, "residual": res}
