"""What a user has this library do, as cases that can be timed and checked.

``listed()`` are the fixed cases, ``draw(rng)`` gives one more of the same
ranges, ``prepare`` makes what a user's program holds before the call (data,
plan, problem, states, output buffers), ``run`` is one pass through the public
entry points, ``work`` the bytes and operations a pass cannot do without and
``exact`` the outputs in 64 bits, from plain torch.

Kinds of cases:

project   pet_forward and pet_back of one subset (or of all views)
steps     updates of one method on one state: ``State.epoch`` (no objectives) or
          ``State.run`` with the objective every so many updates; single
          slices, slice stacks and multi-ring volumes
methods   OSEM, SVREM, SAGA and SVRG at once, a stream each (``State.run``)
batch     a few updates of many uneven reconstructions (``Batch.epoch``)
recon     a served reconstruction from new counts: problem update, warm start,
          state reset, epochs with their objectives
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2106_03172_gb300 import petvr
from paper_2106_03172_gb300.phantoms import (Geometry, Workload, batched_workloads, make_data, subset_sequence)

METHODS = ("osem", "svrem", "saga", "svrg")
# step sizes and anchor periods of the named workloads
ALPHA = {"osem": 1.0, "svrem": 0.7, "saga": 1.0, "svrg": 2.0, "sem": 1.0}
DECAY = {"sem": 0.001}


def _case(name, kind, **kw):
    base = dict(name=name, kind=kind, nx=64, ny=64, views=60, bins=91, pixel_mm=2.0, bin_mm=2.0, nz=1, rings=0,
                ring_mm=0.0, radius_mm=0.0, slice_mm=0.0, subsets=6, counts=1e5, bg=0.1, bg_array=False, beta=0.01,
                potential="quadratic", delta=1.0, ellipses=8, method="osem", table="fp32", eta=1, updates=6,
                objective_every=0, subset=0, members=0)
    base.update(kw)
    return base


def listed():
    c256 = dict(nx=256, ny=256, views=180, bins=367, subsets=21, counts=1e7, beta=0.005, ellipses=20)
    return [
        # the smallest call: one subset's projections of the small 64^2 configuration (launches and latency)
        _case("project_64", "project", subset=2),
        # projections of all views at the 256^2 configuration (an application's own loop over the full data)
        _case("project_all_256", "project", subset=-1, **c256),
        # one epoch of the small configuration, epoch call by epoch call
        _case("osem_64", "steps"),
        # one SAGA epoch of the 256^2 configuration: the single-state chain of subset updates
        _case("saga_256", "steps", method="saga", updates=21, **c256),
        # two SVREM epochs of the 256^2 configuration with anchors and objectives in one call
        _case("svrem_256", "steps", method="svrem", updates=42, objective_every=21, **c256),
        # odd sizes: non-square image, even bin count, bins finer than pixels, Huber penalty, background array
        _case("svrg_odd", "steps", method="svrg", nx=201, ny=147, views=131, bins=250, pixel_mm=1.7, bin_mm=1.4,
              subsets=7, counts=2e6, bg_array=True, beta=0.01, potential="huber", delta=2.0, eta=2, updates=28,
              objective_every=7, ellipses=12),
        # the headline step: the four methods side by side on four streams, objectives after every epoch
        _case("methods_256", "methods", updates=84, objective_every=21, eta=1, **c256),
        # uneven reconstructions advanced together, 3 updates a tick as the batch server does, BF16 tables
        _case("batch_mixed", "batch", members=24, updates=3, method="saga", table="bf16"),
        # the 47-slice stack: two SVRG epochs from an anchor, objective after each
        _case("stack_47", "steps", method="svrg", nx=128, ny=128, views=252, bins=344,
              bin_mm=math.sqrt(2.0) * 128 * 2.0 / 344, nz=47, subsets=14, counts=5e8, bg=0.15, beta=0.002, eta=2,
              updates=28, objective_every=14, ellipses=10),
        # the two-ring volume, log-cosh penalty: an SVREM epoch with its anchor and objective
        _case("ring2_128", "steps", method="svrem", nx=128, ny=128, views=280, bins=183, nz=3, rings=2, ring_mm=4.0,
              radius_mm=400.0, slice_mm=2.0, subsets=20, counts=1e7, beta=0.005, potential="logcosh", eta=3,
              updates=20, objective_every=20, ellipses=12),
        # the largest request of the serving stream from its counts: warm start, reset (table fill), an epoch
        _case("recon_512", "recon", nx=512, ny=512, views=720, bins=733, subsets=12, counts=1e7, beta=0.005,
              method="saga", updates=12, objective_every=12, ellipses=12),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "single", "single", "single", "stack", "ring", "batch", "recon"])
    if kind == "batch":
        return _nameless(_case("", "batch", members=rng.randint(4, 24), updates=rng.randint(2, 4), method="saga",
                               table="bf16", subset=rng.randint(0, 10 ** 6)))
    hi = {"project": 512, "single": 320, "stack": 128, "ring": 128, "recon": 400}[kind]
    nx = _spread(rng, 40, hi)
    ny = nx if rng.random() < 0.5 else max(32, int(nx * rng.uniform(0.7, 1.0)))
    bin_mm = rng.choice([2.0, 2.0, 1.3, 2.6])
    views = max(24, int(nx * rng.uniform(0.6, 1.3)))
    bins = int(1.43 * nx * 2.0 / bin_mm) + rng.randint(0, 1)
    kw = dict(nx=nx, ny=ny, views=views, bins=bins, bin_mm=bin_mm, subsets=rng.randint(4, min(21, views // 4)),
              counts=10.0 ** rng.uniform(2.5, 3.5) * nx, beta=rng.choice([0.002, 0.005, 0.01]),
              bg_array=rng.random() < 0.3, potential=rng.choice(["quadratic", "quadratic", "huber", "logcosh"]),
              ellipses=rng.randint(6, 16))
    if kind == "project":
        kw["subset"] = rng.choice([-1, rng.randint(0, kw["subsets"] - 1)])
        return _nameless(_case("", "project", **kw))
    kw["method"] = rng.choice(["osem", "svrem", "saga", "svrg", "sem"])
    kw["eta"] = rng.randint(1, 2)
    if kind == "recon":
        kw.update(method=rng.choice(["svrem", "saga"]), bg_array=False, potential="quadratic",
                  updates=kw["subsets"], objective_every=kw["subsets"])
        return _nameless(_case("", "recon", **kw))
    if kind == "stack":
        kw.update(nz=_spread(rng, 3, 64), counts=kw["counts"] * 10)
    if kind == "ring":
        kw.update(nz=rng.randint(2, 8), rings=rng.randint(2, 3), ring_mm=4.0, radius_mm=400.0, slice_mm=2.0,
                  views=max(24, views // 2))
        kw["subsets"] = min(kw["subsets"], kw["views"] // 4)
    kw["updates"] = kw["subsets"] * rng.randint(1, 2)
    kw["objective_every"] = rng.choice([0, kw["subsets"]])
    return _nameless(_case("", "steps", **kw))


def _nameless(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---- inputs ------------------------------------------------------------------

def _geometry(c):
    return Geometry(c["nx"], c["ny"], c["views"], c["bins"], pixel_mm=c["pixel_mm"], bin_mm=c["bin_mm"], nz=c["nz"],
                    n_rings=c["rings"], ring_mm=c["ring_mm"], radius_mm=c["radius_mm"], slice_mm=c["slice_mm"])


def _workload(c):
    return Workload("case", _geometry(c), n_subsets=c["subsets"], counts=c["counts"], bg_frac=c["bg"],
                    beta=c["beta"], n_ellipses=c["ellipses"], stack=c["nz"] > 1 and not c["rings"],
                    potential=c["potential"], delta=c["delta"])


def _inputs(work, seed, bg_array):
    """Counts, background and a start image (numpy float32) from the seed alone.

    The start image stands for an iterate: the phantom, flattened towards its
    mean, with a few per cent of noise, positive everywhere."""
    data = make_data(work, seed)
    rng = np.random.default_rng(seed + 77)
    x = data["x_true"]
    img = 0.7 * x + 0.3 * float(x.mean()) + 1e-3 * float(x.max())
    img = (img * rng.uniform(0.95, 1.05, size=x.shape)).astype(np.float32)
    bg = None
    if bg_array:
        bg = (data["w"] * rng.uniform(0.8, 1.2, size=data["g"].shape)).astype(np.float32)
    return data["g"], np.float32(data["w"]), bg, img


def _members(c):
    return batched_workloads(c["subset"], c["members"])


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a).ravel()).cuda()


def _sequence(c, n, seed):
    return [int(t) for t in subset_sequence(1000 + seed, c["subsets"], n)]


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        states, seqs, keep, plans = [], [], [], {}
        for i, work in enumerate(_members(c)):
            g, w, bg, img = _inputs(work, seed + i, False)
            key = (work.geometry, work.n_subsets)
            if key not in plans:
                plans[key] = petvr.Plan(*key)
            prob = petvr.Problem(plans[key], _cuda(g), None, float(w), work.beta)
            states.append(petvr.State(prob, c["method"], _cuda(img), table=c["table"]))
            seqs.append([int(t) for t in subset_sequence(2000 + seed + i, work.n_subsets, c["updates"])])
            keep.append(prob)
        n = len(states)
        return {"case": c, "batch": petvr.Batch(states), "states": states, "seqs": seqs, "alphas": [1.0] * n,
                "etas": [1] * n, "keep": keep}
    work = _workload(c)
    g, w, bg, img = _inputs(work, seed, c["bg_array"])
    plan = petvr.Plan(work.geometry, work.n_subsets)
    s = {"case": c, "plan": plan, "bg": None if bg is None else _cuda(bg), "w": 0.0 if bg is not None else float(w)}
    if c["kind"] == "project":
        rng = np.random.default_rng(seed + 5)
        n = plan.subset_lines(c["subset"]) if c["subset"] >= 0 else c["views"] * c["bins"] * max(1, c["rings"]) ** 2
        s["img"] = _cuda(img)
        s["ratio"] = _cuda(rng.uniform(0.7, 1.3, size=n * (1 if c["rings"] else c["nz"])).astype(np.float32))
        s["bg"], s["w"] = None, float(w)
        s["sino"], s["back"] = torch.empty_like(s["ratio"]), torch.empty_like(s["img"])
        return s
    s["counts"] = _cuda(g)
    s["prob"] = petvr.Problem(plan, s["counts"], s["bg"], s["w"], work.beta, potential=work.potential,
                              delta=work.delta)
    methods = METHODS if c["kind"] == "methods" else (c["method"],)
    s["imgs"] = [_cuda(img) for _ in methods]
    s["states"] = [petvr.State(s["prob"], m, i, table=c["table"]) for m, i in zip(methods, s["imgs"])]
    points = c["updates"] // c["objective_every"] if c["objective_every"] else 0
    s["phis"] = [torch.zeros(points, 3, dtype=torch.float64, device="cuda") for _ in methods] if points else []
    s["seqs"] = [_sequence(c, c["updates"], seed + 13 * k) for k in range(len(methods))]
    s["methods"] = methods
    if c["kind"] == "methods":
        s["streams"] = [torch.cuda.Stream() for _ in methods]
    return s


# ---- one pass ----------------------------------------------------------------

def run(state):
    s, c = state, state["case"]
    if c["kind"] == "project":
        petvr.pet_forward(s["plan"].handle, s["img"], s["bg"], s["w"], c["subset"], s["sino"])
        petvr.pet_back(s["plan"].handle, s["ratio"], c["subset"], s["back"])
        return s["sino"], s["back"]
    if c["kind"] == "batch":
        s["batch"].epoch(s["seqs"], s["alphas"], s["etas"])
        return [st.img for st in s["states"]]
    if c["kind"] == "methods":
        main = torch.cuda.current_stream()
        for stream in s["streams"]:
            stream.wait_stream(main)
        for k, m in enumerate(s["methods"]):
            s["states"][k].run(s["seqs"][k], alpha=ALPHA[m], eta=2 if m == "svrg" else 1,
                               objective_every=c["objective_every"], phi=s["phis"][k], stream=s["streams"][k])
        for stream in s["streams"]:
            main.wait_stream(stream)
        return s["imgs"], s["phis"]
    m, st = c["method"], s["states"][0]
    if c["kind"] == "recon":
        petvr.pet_problem_update(s["prob"].handle, s["counts"], s["bg"], s["w"])
        petvr.pet_warm_start(s["prob"].handle, s["imgs"][0])
        st.reset()
    if c["objective_every"]:
        st.run(s["seqs"][0], alpha=ALPHA[m], decay=DECAY.get(m, 0.0), eta=c["eta"],
               objective_every=c["objective_every"], phi=s["phis"][0])
        return s["imgs"][0], s["phis"][0]
    st.epoch(s["seqs"][0], alpha=ALPHA[m], eta=c["eta"], decay=DECAY.get(m, 0.0))
    return s["imgs"][0]


# ---- work --------------------------------------------------------------------

def _nnz(geom, views):
    """Nonzeros of the system rows of `views` views over half a turn: a view's
    rays cross a pixel (|cos| + |sin|) pixel/bin times on average, 4/pi over
    the views; a line of a multi-ring scanner meets its own layers only."""
    per = geom.n_pixels * 4.0 / math.pi * geom.pixel_mm / geom.ds
    return per * views * geom.n_pairs


def _update_work(geom, ns, method, table, updates):
    views = geom.n_angles / ns
    pixels = geom.n_pixels * (geom.nz if geom.nz > 1 else 1)
    per_pixel = {"osem": 12, "sem": 20, "svrem": 32, "saga": 28 if table == "bf16" else 32, "svrg": 20}[method]
    lines = views * geom.n_bins * geom.n_pairs
    return updates * (4.0 * lines + per_pixel * pixels), updates * 4.0 * _nnz(geom, views)


def work(case):
    c = case
    if c["kind"] == "batch":
        b = f = 0.0
        for w in _members(c):
            x, y = _update_work(w.geometry, w.n_subsets, c["method"], c["table"], c["updates"])
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    geom = _geometry(c)
    pixels = geom.n_pixels * geom.nz
    full_lines = geom.n_rays * geom.n_pairs
    if c["kind"] == "project":
        part = 1.0 if c["subset"] < 0 else 1.0 / c["subsets"]
        return {"bytes": 8.0 * pixels + 8.0 * full_lines * part,
                "flops": 4.0 * _nnz(geom, geom.n_angles * part)}
    b = f = 0.0
    for m in METHODS if c["kind"] == "methods" else (c["method"],):
        eta = {"svrg": 2, "svrem": 1}.get(m, 1) if c["kind"] == "methods" else c["eta"]
        x, y = _update_work(geom, c["subsets"], m, c["table"], c["updates"])
        # a full pass is a forward and a back projection of every view; an objective a forward
        full = math.ceil(c["updates"] / (eta * c["subsets"])) if m in ("svrem", "svrg") else 0
        points = c["updates"] // c["objective_every"] if c["objective_every"] else 0
        if c["kind"] == "recon":
            x2, y2 = _update_work(geom, c["subsets"], "osem", c["table"], c["subsets"])
            x, y = x + x2 + 8.0 * full_lines, y + y2
            full += 1 if m == "saga" else 0
        shared = min(points, max(0, full - 1))     # an objective's forward serves the next anchor
        x += full * (4.0 * full_lines + 4.0 * pixels * (1 + c["subsets"])) + (points - shared) * 4.0 * (
            full_lines + pixels)
        y += full * 4.0 * _nnz(geom, geom.n_angles) + (points - shared) * 2.0 * _nnz(geom, geom.n_angles)
        b, f = b + x, f + y
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits -----------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _snap(v):
    return float(round(v)) if abs(v - round(v)) < 1e-12 else v


class _Exact:
    """The model in 64 bits: Siddon's intersection lengths enumerated along
    each view's major image axis, and the methods' updates."""

    def __init__(self, work):
        self.g, self.ns, self.dev = work.geometry, work.n_subsets, _device()
        g = self.g
        self.vol = (g.ny * g.nx, g.nz)                 # pixels x (slices or layers)
        self.sens_t = [self.back(t, torch.ones((g.n_bins * len(self.views(t)), self.lines_z()), dtype=torch.float64,
                                               device=self.dev)) for t in range(self.ns)]
        self.sens = sum(self.sens_t)

    def lines_z(self):
        return self.g.n_pairs

    def views(self, t):
        return range(self.g.n_angles) if t < 0 else range(t, self.g.n_angles, self.ns)

    def _view(self, i):
        """Pixel indices and weights, each (bins, bands, 2), of view i, and
        for a multi-ring scanner the piece's share of every layer."""
        g, f8 = self.g, dict(dtype=torch.float64, device=self.dev)
        th = i * math.pi / g.n_angles
        co, si = _snap(math.cos(th)), _snap(math.sin(th))
        col = abs(co) < abs(si)
        cm, cn = (si, co) if col else (co, si)
        n_major, n_minor = (g.nx, g.ny) if col else (g.ny, g.nx)
        s = (torch.arange(g.n_bins, **f8) - 0.5 * (g.n_bins - 1)) * g.ds
        k = torch.arange(n_major + 1, **f8) - 0.5 * n_major
        # relative to the pixel edge next to the centre, so that a ray on a grid line falls on an integer
        u = (s / (cm * g.pixel_mm) + 0.5 * (n_minor % 2))[:, None] - k[None, :] * (cn / cm)
        lo, hi = torch.minimum(u[:, :-1], u[:, 1:]), torch.maximum(u[:, :-1], u[:, 1:])
        fl = torch.floor(lo)
        length = g.pixel_mm / abs(cm)
        share = torch.where(hi <= fl + 1, torch.ones_like(lo), (fl + 1 - lo) / max(abs(cn / cm), 1e-300))
        w = torch.stack([share, 1 - share], -1) * length
        m = torch.stack([fl, fl + 1], -1).long() + n_minor // 2
        ok = (m >= 0) & (m < n_minor)
        kk = torch.arange(n_major, device=self.dev)[None, :, None]
        idx = torch.where(ok, m * g.nx + kk if col else kk * g.nx + m, torch.zeros_like(m))
        w = torch.where(ok, w, torch.zeros_like(w))
        if not g.multiring:
            return idx, w, None
        # axial: arc length along (-sin, cos) at band boundaries, linear in k
        t = (s[:, None] * co / si - k[None, :] * g.pixel_mm / si) if col else (
            -s[:, None] * si / co + k[None, :] * g.pixel_mm / co)
        z = (torch.arange(g.n_rings, **f8) - 0.5 * (g.n_rings - 1)) * g.ring_mm
        z1, z2 = [v.reshape(-1) for v in torch.meshgrid(z, z, indexing="ij")]
        kappa = (z2 - z1)[None, :] / (2.0 * torch.sqrt(g.radius_mm ** 2 - s * s))[:, None]      # bins x pairs
        zeta = ((0.5 * (z1 + z2))[None, None, :] + kappa[:, None, :] * t[:, :, None]) / g.slice_mm + 0.5 * g.nz
        first_lower = cn / cm < 0                     # u grows with k: pixel fl is met first
        a = torch.where(torch.tensor(first_lower, device=self.dev), share, 1 - share)[..., None]
        z0, ze = zeta[:, :-1], zeta[:, 1:]
        mid = z0 + a * (ze - z0)
        lower, upper = ((z0, mid), (mid, ze)) if first_lower else ((mid, ze), (z0, mid))
        za = torch.stack([lower[0], upper[0]], 2)     # bins x bands x 2 x pairs
        zb = torch.stack([lower[1], upper[1]], 2)
        zl, zh = torch.minimum(za, zb)[..., None], torch.maximum(za, zb)[..., None]
        iz = torch.arange(g.nz, **f8)
        span = (zh - zl)
        over = (torch.minimum(zh, iz + 1) - torch.maximum(zl, iz)).clamp(min=0.0)
        lay = torch.where(span > 1e-12, over / span.clamp(min=1e-300), (torch.floor(0.5 * (zl + zh)) == iz).double())
        return idx, w, lay * torch.sqrt(1 + kappa * kappa)[:, None, None, :, None]

    def forward(self, t, f):
        out = []
        for i in self.views(t):
            idx, w, lay = self._view(i)
            v = f[idx]                                # bins x bands x 2 x z
            if lay is None:
                out.append((v * w[..., None]).sum((1, 2)))
            else:
                out.append(torch.einsum("jkbz,jkbpz,jkb->jp", v, lay, w))
        return torch.cat(out)

    def back(self, t, r):
        g = self.g
        out = torch.zeros(self.vol, dtype=torch.float64, device=self.dev)
        for q, i in enumerate(self.views(t)):
            idx, w, lay = self._view(i)
            rv = r[q * g.n_bins:(q + 1) * g.n_bins]
            if lay is None:
                v = w[..., None] * rv[:, None, None, :]
            else:
                v = torch.einsum("jkb,jkbpz,jp->jkbz", w, lay, rv)
            out.index_add_(0, idx.reshape(-1), v.reshape(-1, g.nz))
        return out

    def bind(self, counts, w, bg, beta, pot, delta):
        n = self.g.n_angles * self.g.n_bins
        f8 = lambda a: torch.from_numpy(np.asarray(a, dtype=np.float64)).reshape(n, -1).to(self.dev)  # noqa: E731
        self.counts = f8(counts)
        self.w = f8(bg) if bg is not None else torch.full_like(self.counts, float(w))
        self.beta, self.pot, self.delta = float(np.float32(beta)), pot, float(np.float32(delta))

    def rows(self, x, t):
        return x.reshape(self.g.n_angles, self.g.n_bins, -1)[list(self.views(t))].reshape(-1, x.shape[-1])

    def ratio(self, t, f):
        y = self.forward(t, f) + self.rows(self.w, t)
        return torch.where(y != 0, self.rows(self.counts, t) / torch.where(y != 0, y, torch.ones_like(y)),
                           torch.zeros_like(y))

    def stat(self, t, f):
        return self.back(t, self.ratio(t, f))

    def _pairs(self, f):
        """(own index slices, neighbour index slices) of every ordered neighbour pair, on (ny, nx, z)."""
        a, b = slice(1, None), slice(None, -1)
        dims = (0, 1, 2) if self.g.multiring else (0, 1)
        for d in dims:
            for own, other in ((a, b), (b, a)):
                i, j = [slice(None)] * 3, [slice(None)] * 3
                i[d], j[d] = own, other
                yield tuple(i), tuple(j)

    def _rho(self, t):
        d = self.delta
        if self.pot == "huber":
            return torch.where(t.abs() <= d, 0.5 * t * t, d * t.abs() - 0.5 * d * d)
        if self.pot == "logcosh":
            u = (t / d).abs()
            return d * d * (u + torch.log1p(torch.exp(-2 * u)) - math.log(2.0))
        return 0.5 * t * t

    def _curve(self, t):
        d = self.delta
        if self.pot == "huber":
            return torch.where(t.abs() <= d, torch.ones_like(t), d / t.abs().clamp(min=1e-300))
        if self.pot == "logcosh":
            return torch.where(t != 0, d * torch.tanh(t / d) / torch.where(t != 0, t, torch.ones_like(t)),
                               torch.ones_like(t))
        return torch.ones_like(t)

    def stencil(self, f):
        """Sum of the surrogate weights, of weights times neighbours, and the penalty gradient."""
        v = f.reshape(self.g.ny, self.g.nx, -1)
        cnt, tot, grad = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
        for i, j in self._pairs(v):
            t = v[i] - v[j]
            c = self._curve(t)
            cnt[i] += c
            tot[i] += c * v[j]
            grad[i] += c * t
        return cnt.reshape(f.shape), tot.reshape(f.shape), grad.reshape(f.shape)

    def penalty(self, f):
        v = f.reshape(self.g.ny, self.g.nx, -1)
        return 0.5 * sum(self._rho(v[i] - v[j]).sum() for i, j in self._pairs(v))

    def objective(self, f):
        y = self.forward(-1, f) + self.w
        ll = torch.where(self.counts > 0, self.counts * torch.log(y.clamp(min=1e-300)), torch.zeros_like(y)) - y
        a, r = ll.sum(), self.penalty(f)
        return torch.stack([a - self.beta * r, a, r])

    def root(self, f, a, S, beta):
        """Nonnegative root of a/x - 2 b x + c = 0 (the surrogate M-step); 0 where S <= 0 or a <= 0."""
        cnt, tot, _ = self.stencil(f)
        b, c = beta * cnt, beta * (f * cnt + tot) - S
        d = torch.sqrt(c * c + 8 * a.clamp(min=0) * b)
        x = torch.where(c <= 0, 2 * a / (d - c).clamp(min=1e-300), (c + d) / (4 * b).clamp(min=1e-300))
        return torch.where((S > 0) & (a > 0), x, torch.zeros_like(x))

    def grad_t(self, t, f):
        return self.stat(t, f) - self.sens_t[t] - self.beta / self.ns * self.stencil(f)[2]

    def warm_start(self):
        z = self.counts.shape[1]
        tot = (self.counts - self.w).clamp(min=0).sum(0)
        f = (tot / self.sens[:, :1].sum() if z > 1 else tot / self.sens.sum()).expand(self.vol).clone()
        keep, self.beta = self.beta, 0.0
        for t in range(self.ns):
            f = self.root(f, f * self.stat(t, f), self.sens_t[t], 0.0)
        self.beta = keep
        return f

    def steps(self, method, f, seq, alpha, decay, eta, every):
        ns, beta, points = self.ns, self.beta, []
        alpha, decay = float(np.float32(alpha)), float(np.float32(decay))
        d = torch.where(self.sens > 0, ns * f / self.sens.clamp(min=1e-300), torch.zeros_like(f))
        if method == "saga":
            table = [self.grad_t(t, f) for t in range(ns)]
            mean = sum(table) / ns
        s_hat = None
        for k, t in enumerate(seq):
            if method in ("svrem", "svrg") and k % (eta * ns) == 0:
                f_anc, B = f, [self.stat(q, f) for q in range(ns)]
                total = sum(B)
                if method == "svrem" and s_hat is None:
                    s_hat = f * total
            if method == "osem":
                f = self.root(f, f * self.stat(t, f), self.sens_t[t], beta / ns)
            elif method == "sem":
                if s_hat is None:
                    s_hat = f * self.stat(-1, f)
                a = float(np.float32(alpha / (decay * k + 1.0)))
                s_hat = (1 - a) * s_hat + a * ns * f * self.stat(t, f)
                f = self.root(f, s_hat, self.sens, beta)
            elif method == "svrem":
                tau = ns * f * self.stat(t, f) - ns * f_anc * B[t] + f_anc * total
                s_hat = (1 - alpha) * s_hat + alpha * tau
                f = self.root(f, s_hat, self.sens, beta)
            elif method == "saga":
                q = self.grad_t(t, f)
                f = (f + alpha * d * (q - table[t] + mean)).clamp(min=0)
                mean = mean + (q - table[t]) / ns
                table[t] = q
            else:
                step = (self.stat(t, f) - B[t] - beta / ns * self.stencil(f)[2] + (total - self.sens) / ns)
                f = (f + alpha * d * step).clamp(min=0)
            if every and (k + 1) % every == 0:
                points.append(self.objective(f))
        return f, points


def exact(case, seed):
    c = case

    def flat(f):
        return f.reshape(-1).cpu()

    if c["kind"] == "batch":
        out = []
        for i, work in enumerate(_members(c)):
            g, w, bg, img = _inputs(work, seed + i, False)
            m = _Exact(work)
            m.bind(g, w, None, work.beta, "quadratic", 1.0)
            seq = [int(t) for t in subset_sequence(2000 + seed + i, work.n_subsets, c["updates"])]
            f0 = torch.from_numpy(img.astype(np.float64)).reshape(m.vol).to(m.dev)
            out.append(flat(m.steps(c["method"], f0, seq, 1.0, 0.0, 1, 0)[0]))
        return out
    work = _workload(c)
    g, w, bg, img = _inputs(work, seed, c["bg_array"])
    m = _Exact(work)
    f0 = torch.from_numpy(img.astype(np.float64)).reshape(m.vol).to(m.dev)
    if c["kind"] == "project":
        t = c["subset"]
        rng = np.random.default_rng(seed + 5)
        rows = len(m.views(t)) * c["bins"]
        r = rng.uniform(0.7, 1.3, size=rows * m.lines_z()).astype(np.float32).astype(np.float64)
        r = torch.from_numpy(r).reshape(rows, -1).to(m.dev)
        return flat(m.forward(t, f0) + float(w)), flat(m.back(t, r))
    m.bind(g, w, bg, work.beta, work.potential, work.delta)
    imgs, phis = [], []
    for k, name in enumerate(METHODS if c["kind"] == "methods" else (c["method"],)):
        f = m.warm_start() if c["kind"] == "recon" else f0
        eta = (2 if name == "svrg" else 1) if c["kind"] == "methods" else c["eta"]
        f, points = m.steps(name, f, _sequence(c, c["updates"], seed + 13 * k), ALPHA[name], DECAY.get(name, 0.0),
                            eta, c["objective_every"])
        imgs.append(flat(f))
        if points:
            phis.append(torch.stack(points).cpu())
    if c["kind"] == "methods":
        return imgs, phis
    return (imgs[0], phis[0]) if phis else imgs[0]
