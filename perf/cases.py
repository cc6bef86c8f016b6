"""The work that a user of this library has it do, case by case: what is timed when its speed is measured.

A case names one or several acquisition geometries (image side n, detectors on an arc, time samples, angular nodes), the
image storage type and the call: the operators by themselves, one iteration of each solver, the gradient that a
training loop takes, the TV term, and one whole solver run.  Everything goes through :class:`PatPlan`,
:mod:`paper_2604_19176_gb300.graphs` and :mod:`paper_2604_19176_gb300.recon`, with the plan that a program keeps
for its geometry (default options) made in ``prepare``.

Images are vessel-like tubes and Gaussian blobs, data are the pulses that a few point sources would send to each
detector, with noise: both are drawn on the GPU from the seed alone.

``exact`` evaluates the same discrete operators in FP64 with plain tensor arithmetic (bilinear samples on the
circles, closed-form Abel weights).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan
from paper_2604_19176_gb300.graphs import GraphedOperator
from paper_2604_19176_gb300.recon import pat_apply, tv_reconstruct, tv_value

T_MAX = 2.0
EPS = 1e-3       # smoothing of the TV term
LAM = 1e-3       # TV weight of the variational solvers
DIP_LAM = 1e-4   # TV weight of the training loss

# Largest (detector, radius, angle) count of a drawn case, over all its images
MOST_DRAWN = 600_000_000


def _case(name, call, n, n_det, degrees, n_t, n_angles, batch=1, dtype="float32", **more):
    c = {"call": call, "n": n, "n_det": n_det, "degrees": degrees, "n_t": n_t, "n_angles": n_angles, "batch": batch,
         "dtype": dtype, **more}
    return {"name": name, **c} if name else c


def listed():
    return [
        # The smallest problem: 64^2, full ring, one operator call; latency and launches count
        _case("forward_64", "forward", 64, 64, 360.0, 128, 128),
        # The limited-view 256^2 problem (128 detectors on a half ring): A and A^T as a user's own solver calls them
        _case("forward_256", "forward", 256, 128, 180.0, 512, 512),
        _case("adjoint_256", "adjoint", 256, 128, 180.0, 512, 512),
        # ... one fused projected-gradient iteration of the TV reconstruction, with the benchmark's arguments
        _case("tv_step_256", "tv_step", 256, 128, 180.0, 512, 512),
        # ... the loss and the image gradient that the deep-image-prior loop asks for on every iteration
        _case("loss_grad_256", "loss_grad", 256, 128, 180.0, 512, 512),
        # ... a whole short TV reconstruction: separate calls, the relative change read back after each iteration
        _case("tv_run_256", "tv_run", 256, 128, 180.0, 512, 512, iters=10),
        # Odd sizes throughout: image, detectors, times, nodes and arc off every round number, three images
        _case("pair_ragged", "pair", 100, 37, 118.125, 301, 203, batch=3),
        # The next size up of the limited-view problem
        _case("adjoint_512", "adjoint", 512, 256, 180.0, 1024, 1024),
        # The TV term by itself (value and gradient) on a batch of images
        _case("tv_grad_512x4", "tv_grad", 512, 64, 180.0, 256, 512, batch=4),
        # The experimental ring (256 detectors on 270 degrees, 2030 times): one primal-dual iteration with the
        # sums that its stop rule reads
        _case("pdhg_step_760", "pdhg_step", 760, 256, 270.0, 2030, 1520),
        # 64 measurement sets of uneven size, forward and adjoint replayed from one graph
        _case("graph_uneven_64", "graph_pair", 384, 512, 360.0, 1024, 768, batch=64, uneven=4),
        # The precision study: eight 1024^2 images stored in BF16, forward and adjoint
        _case("pair_1024x8_bf16", "pair", 1024, 512, 270.0, 2048, 2048, batch=8, dtype="bfloat16"),
    ]


def _spread(rng, lo, hi, step=1):
    """A whole number between lo and hi, spread over its logarithm, a multiple of step."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    while True:
        call = rng.choice(["forward", "adjoint", "pair", "graph_pair", "tv_step", "pdhg_step", "loss_grad", "tv_grad",
                           "tv_run"])
        dtype = "bfloat16" if call in ("forward", "adjoint", "pair") and rng.random() < 0.3 else "float32"
        n = _spread(rng, 64, 1024, 8 if dtype == "bfloat16" else 4)
        n_det = _spread(rng, 16, 512)
        n_t = max(64, min(2048, int(n * rng.uniform(1.0, 3.0))))
        n_angles = max(64, int(n * rng.uniform(1.5, 2.5))) if rng.random() < 0.5 else 2 * n
        batch = rng.choice([1, 1, 1, 2, 3, 4, 8])
        degrees = rng.choice([90.0, 180.0, 270.0, 360.0, round(rng.uniform(45.0, 360.0), 2)])
        c = _case(None, call, n, n_det, degrees, n_t, n_angles, batch, dtype)
        if call == "tv_run":
            c["iters"] = rng.randint(4, 12)
        if call == "graph_pair" and rng.random() < 0.5:
            c["uneven"] = rng.randint(1, 10**6)
        if sum(g.n_det * g.n_r * g.n_angles for g in geometries(c)) * c.get("iters", 1) <= MOST_DRAWN:
            return c


def geometries(case):
    if "uneven" in case:
        # sizes up to the case's own, drawn per image as in the 64-instance workload
        rng = np.random.default_rng(case["uneven"])
        out = []
        for _ in range(case["batch"]):
            n = max(64, int(case["n"] * rng.choice([128, 192, 256, 384]) / 384) // 4 * 4)
            deg = float(rng.choice([90.0, 180.0, 270.0, 360.0]))
            nd = max(1, int(case["n_det"] * rng.choice([64, 128, 256, 512]) / 512))
            nt = max(16, int(case["n_t"] * rng.choice([256, 512, 1024]) / 1024))
            out.append(Geometry(n, nd, 0.0, math.radians(deg), nt, T_MAX, 2 * n))
        return out
    g = Geometry(case["n"], case["n_det"], 0.0, math.radians(case["degrees"]), case["n_t"], T_MAX, case["n_angles"])
    return [g] * case["batch"]


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bfloat16" else torch.float32


# -- inputs -------------------------------------------------------------------------------------------------------------

def _phantom(n, rng):
    """Tubes of two to four pixels' width and a few Gaussian blobs inside the unit disk, n x n FP32."""
    x = (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) * (2.0 / n) - 1.0
    X, Y = x[None, :], x[:, None]
    f = torch.zeros(n, n, device="cuda")
    for _ in range(8):
        p = _point(rng, 0.8)
        heading, amp, half = rng.uniform(0, 2 * math.pi), rng.uniform(0.3, 1.0), rng.uniform(1.0, 2.0) * 2.0 / n
        for _ in range(3):
            length = rng.uniform(0.1, 0.4)
            heading += rng.uniform(-math.pi / 4, math.pi / 4)
            ax, ay = length * math.cos(heading), length * math.sin(heading)
            t = (((X - p[0]) * ax + (Y - p[1]) * ay) / (length * length)).clamp(0, 1)
            d = torch.sqrt((X - p[0] - t * ax) ** 2 + (Y - p[1] - t * ay) ** 2)
            f = torch.maximum(f, amp * ((half - d) * (n / 2.0) + 0.5).clamp(0, 1))
            p = (p[0] + ax, p[1] + ay)
    for _ in range(5):
        c, s, a = _point(rng, 0.8), rng.uniform(0.03, 0.1), rng.uniform(0.5, 1.0)
        f = f + a * torch.exp(-((X - c[0]) ** 2 + (Y - c[1]) ** 2) / (s * s))
    return f


def _point(rng, radius):
    r, t = radius * math.sqrt(rng.uniform()), rng.uniform(0, 2 * math.pi)
    return (r * math.cos(t), r * math.sin(t))


def _measured(g, rng, gen):
    """What the detectors of g record of a few small sources: a bipolar pulse at each arrival time, and 1 % noise."""
    th = g.arc_start + (torch.arange(g.n_det, device="cuda", dtype=torch.float32) + 0.5) * (g.arc_span / g.n_det)
    t = (torch.arange(g.n_t, device="cuda", dtype=torch.float32) + 1) * (g.t_max / g.n_t)
    out = torch.zeros(g.n_det, g.n_t, device="cuda")
    for _ in range(6):
        c, s, a = _point(rng, 0.8), rng.uniform(0.02, 0.08), rng.uniform(0.1, 0.5)
        u = (t[None, :] - torch.hypot(torch.cos(th) - c[0], torch.sin(th) - c[1])[:, None]) / s
        out = out - a * u * torch.exp(-u * u)
    return out + 0.01 * 0.3 * torch.randn(out.shape, generator=gen, device="cuda")


def _inputs(case, seed):
    """Packed images f and data g of every instance (FP32), and a generator for what else is drawn."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    geoms = geometries(case)
    f = torch.cat([_phantom(g.n, rng).reshape(-1) for g in geoms])
    g = torch.cat([_measured(g, rng, gen).reshape(-1) for g in geoms])
    return geoms, f, g, gen


def _solver_steps(geoms):
    """A step length below 1 / (||A||^2 + 8) for every geometry: ||A||^2 is about 2 to 4 n_det n_t / n^2 on a half or
    full ring, and larger on a shorter arc."""
    return min(1.0 / (8.0 + 8.0 * max(1.0, math.pi / g.arc_span) * g.n_det * g.n_t / g.n**2) for g in geoms)


def _pdhg_start(case, seed):
    """Inputs and the five variables of a primal-dual run some iterations after its start."""
    geoms, f, g, gen = _inputs(case, seed)
    noise = lambda like, s: s * torch.randn(like.shape, generator=gen, device="cuda")  # noqa: E731
    fbar = (f + noise(f, 0.02)).clamp_min(0)
    y, px, py = 0.1 * g + noise(g, 0.01), noise(f, 0.3 * LAM), noise(f, 0.3 * LAM)
    return geoms, f, fbar, y, px, py, g


def prepare(case, seed):
    call = case["call"]
    if call == "pdhg_step":
        geoms, f, fbar, y, px, py, g = _pdhg_start(case, seed)
        plan = PatPlan(geoms)
        img, dat = plan.image_shape(), plan.data_shape()
        step = math.sqrt(_solver_steps(geoms))
        return {"call": call, "plan": plan, "f": f.reshape(img), "fbar": fbar.reshape(img), "y": y.reshape(dat),
                "px": px.reshape(img), "py": py.reshape(img), "g": g.reshape(dat), "step": step,
                "delta": torch.empty(2 * len(geoms), device="cuda")}
    geoms, f, g, _ = _inputs(case, seed)
    plan = PatPlan(geoms, image_dtype=_dtype(case))
    f, g = f.reshape(plan.image_shape()).to(_dtype(case)), g.reshape(plan.data_shape())
    s = {"call": call, "plan": plan, "f": f, "g": g}
    if call == "graph_pair":
        s["op"] = GraphedOperator(plan)
        s["op"].f_in.copy_(f)
        s["op"].g_in.copy_(g)
    elif call == "tv_step":
        s["out"], s["tau"] = torch.empty_like(f), _solver_steps(geoms)
    elif call == "tv_run":
        s["iters"], s["tau"] = case["iters"], _solver_steps(geoms)
    elif call == "loss_grad":
        s["f"] = f.requires_grad_()
    return s


def run(s):
    call, plan = s["call"], s["plan"]
    if call == "forward":
        return plan.forward(s["f"])
    if call == "adjoint":
        return plan.adjoint(s["g"])
    if call == "pair":
        return plan.forward(s["f"]), plan.adjoint(s["g"])
    if call == "graph_pair":
        s["op"].replay()
        return s["op"].g_out, s["op"].f_out
    if call == "tv_step":
        plan.tv_step(s["f"], s["out"], s["g"], s["tau"], LAM, EPS)
        return s["out"]
    if call == "pdhg_step":
        plan.pdhg_step(s["f"], s["fbar"], s["y"], s["px"], s["py"], s["g"], s["step"], s["step"], LAM,
                       delta=s["delta"])
        return {k: s[k] for k in ("f", "fbar", "y", "px", "py", "delta")}
    if call == "tv_grad":
        return plan.tv_grad(s["f"], EPS)
    if call == "tv_run":
        return tv_reconstruct(plan, s["g"], LAM, EPS, iters=s["iters"], tau=s["tau"])
    f = s["f"]
    f.grad = None
    r = pat_apply(f, plan) - s["g"]
    loss = (r * r).sum() + DIP_LAM * tv_value(f, plan, EPS).sum()
    loss.backward()
    return loss.detach(), f.grad


# -- the work that a pass cannot do without -----------------------------------------------------------------------------

def _samples(g):
    """About how many (detector, radius, angle) samples of g fall on its image (a part of them counted)."""
    j = np.unique(np.linspace(0, g.n_det - 1, min(g.n_det, 12)).astype(int))
    m = np.unique(np.linspace(0, g.n_r - 1, min(g.n_r, 96)).astype(int))
    q = np.linspace(0, 2 * math.pi, 192, endpoint=False)
    th = g.arc_start + (j + 0.5) * g.arc_span / g.n_det
    r = m * g.t_max / g.n_t
    x = np.cos(th)[:, None, None] + r[None, :, None] * np.cos(q)
    y = np.sin(th)[:, None, None] + r[None, :, None] * np.sin(q)
    share = np.mean((np.abs(x) <= 1 + 1.0 / g.n) & (np.abs(y) <= 1 + 1.0 / g.n))
    return float(share) * g.n_det * g.n_r * g.n_angles


def work(case):
    geoms = geometries(case)
    size = 2 if case["dtype"] == "bfloat16" else 4
    pixels = sum(g.n * g.n for g in geoms)
    data = sum(g.n_det * g.n_t for g in geoms)
    call = case["call"]
    if call == "tv_grad":
        return {"bytes": 8 * pixels + 4 * len(geoms), "flops": 20 * pixels}
    # one operator: a bilinear sample (8), then the triangle of the Abel matrix, a multiply and an add each
    op = sum(8 * _samples(g) for g in geoms) + sum(float(g.n_det) * g.n_t * (g.n_t + 5) for g in geoms)
    if call in ("forward", "adjoint"):
        return {"bytes": size * pixels + 4 * data, "flops": op}
    if call in ("pair", "graph_pair"):
        return {"bytes": 2 * (size * pixels + 4 * data), "flops": 2 * op}
    if call == "tv_step":
        return {"bytes": 8 * pixels + 4 * data, "flops": 2 * op + 26 * pixels}
    if call == "pdhg_step":
        return {"bytes": 32 * pixels + 12 * data, "flops": 2 * op + 30 * pixels + 5 * data}
    if call == "loss_grad":
        return {"bytes": 8 * pixels + 4 * data, "flops": 2 * op + 24 * pixels + 4 * data}
    return {"bytes": 4 * pixels + 4 * data, "flops": case["iters"] * (2 * op + 30 * pixels + 2 * data)}


# -- the same results in FP64 -------------------------------------------------------------------------------------------

def _abel(n_t):
    """Abel matrix P (n_t x (n_t + 2)): exact product integration of the piecewise-linear mean, midpoint derivative."""
    tau = (torch.arange(n_t + 1, dtype=torch.float64, device="cuda") + 0.5)[:, None]
    s = torch.arange(n_t + 1, dtype=torch.float64, device="cuda")[None, :]
    a, b = torch.minimum(s, tau), torch.minimum(s + 1, tau)
    root = lambda r: torch.sqrt(((tau - r) * (tau + r)).clamp_min(0))  # noqa: E731
    i1 = root(a) - root(b)
    i2 = 0.5 * tau * tau * (torch.asin(b / tau) - torch.asin(a / tau)) - 0.5 * (b * root(b) - a * root(a))
    w = torch.zeros(n_t + 1, n_t + 2, dtype=torch.float64, device="cuda")
    w[:, 1:] += i2 - s * i1
    w[:, :-1] += (s + 1) * i1 - i2
    return w[1:] - w[:-1]


class _Operator:
    """A and A^T of `batch` images of one geometry in FP64; images (batch, n, n), data (batch, n_det, n_t)."""

    def __init__(self, g, batch):
        self.g, self.batch, self.P = g, batch, _abel(g.n_t)
        self.per = max(1, 6_000_000 // (g.n_r * g.n_angles))   # detectors at a time
        self.kept = None

    def _chunks(self):
        if self.kept is None:
            made = self._make()
            if self.g.n_det * self.g.n_r * self.g.n_angles > 200_000_000:
                return made
            self.kept = list(made)
        return self.kept

    def _make(self):
        """(detectors, index of (detector, radius), cell index, fractions) of the samples that touch the image."""
        g = self.g
        n, w = g.n, g.n + 2   # one ring of zeros around the image
        d = dict(dtype=torch.float64, device="cuda")
        m = torch.arange(g.n_r, **d) * (g.t_max / g.n_t * n / 2.0)
        q = torch.arange(g.n_angles, **d) * (2.0 * math.pi / g.n_angles)
        for j0 in range(0, g.n_det, self.per):
            j = torch.arange(j0, min(j0 + self.per, g.n_det), **d)
            th = g.arc_start + (j + 0.5) * (g.arc_span / g.n_det)
            x = (torch.cos(th) * (n / 2.0) - 0.5 + n / 2.0)[:, None, None] + m[None, :, None] * torch.cos(q)
            y = (torch.sin(th) * (n / 2.0) - 0.5 + n / 2.0)[:, None, None] + m[None, :, None] * torch.sin(q)
            at = ((x >= -1) & (x < n) & (y >= -1) & (y < n)).reshape(-1).nonzero()[:, 0]
            x, y = x.reshape(-1)[at], y.reshape(-1)[at]
            cx, cy = torch.floor(x), torch.floor(y)
            yield (j0, j0 + len(j), at // g.n_angles, ((cy.long() + 1) * w + cx.long() + 1), x - cx, y - cy)

    @staticmethod
    def _corners(w, cell, a, b):
        yield cell, (1 - a) * (1 - b)
        yield cell + 1, a * (1 - b)
        yield cell + w, (1 - a) * b
        yield cell + w + 1, a * b

    def forward(self, f):
        g, w = self.g, self.g.n + 2
        img = torch.nn.functional.pad(f, (1, 1, 1, 1)).reshape(self.batch, -1).T.contiguous()
        M = torch.empty(g.n_det, g.n_r, self.batch, dtype=torch.float64, device="cuda")
        for j0, j1, at, cell, a, b in self._chunks():
            v = 0
            for c, wt in self._corners(w, cell, a, b):
                v = v + wt[:, None] * img[c]
            row = torch.zeros((j1 - j0) * g.n_r, self.batch, dtype=torch.float64, device="cuda")
            M[j0:j1] = row.index_add_(0, at, v).reshape(j1 - j0, g.n_r, self.batch)
        return torch.einsum("jmb,km->bjk", M, self.P) / g.n_angles

    def adjoint(self, data):
        g, w = self.g, self.g.n + 2
        M = torch.einsum("bjk,km->jmb", data, self.P)
        out = torch.zeros(w * w, self.batch, dtype=torch.float64, device="cuda")
        for j0, j1, at, cell, a, b in self._chunks():
            v = M[j0:j1].reshape(-1, self.batch)[at]
            for c, wt in self._corners(w, cell, a, b):
                out.index_add_(0, c, wt[:, None] * v)
        return out.T.reshape(self.batch, w, w)[:, 1:-1, 1:-1] / g.n_angles


class _Packed:
    """The operators of a plan's packed images and data."""

    def __init__(self, geoms):
        self.geoms, ops = geoms, {}
        if all(g == geoms[0] for g in geoms):
            self.parts = [(_Operator(geoms[0], len(geoms)), len(geoms))]
        else:
            self.parts = [(ops.setdefault(g, _Operator(g, 1)), 1) for g in geoms]

    def _each(self, x, size, shape, fn):
        out, at = [], 0
        for op, b in self.parts:
            k = b * size(op.g)
            out.append(fn(op)(x[at:at + k].reshape(b, *shape(op.g))).reshape(-1))
            op.kept = None if len(self.parts) > 1 else op.kept
            at += k
        return torch.cat(out)

    def forward(self, f):
        return self._each(f, lambda g: g.n * g.n, lambda g: (g.n, g.n), lambda op: op.forward)

    def adjoint(self, d):
        return self._each(d, lambda g: g.n_det * g.n_t, lambda g: (g.n_det, g.n_t), lambda op: op.adjoint)

    def images(self, f):
        at = 0
        for g in self.geoms:
            yield f[at:at + g.n * g.n].reshape(g.n, g.n)
            at += g.n * g.n


def _grad(f):
    dx, dy = torch.zeros_like(f), torch.zeros_like(f)
    dx[:, :-1], dy[:-1] = f[:, 1:] - f[:, :-1], f[1:] - f[:-1]
    return dx, dy


def _grad_t(px, py):
    out = torch.zeros_like(px)
    out[:, :-1] -= px[:, :-1]
    out[:, 1:] += px[:, :-1]
    out[:-1] -= py[:-1]
    out[1:] += py[:-1]
    return out


def _tv(op, f):
    """TV value of every image and the packed gradient."""
    vals, grads = [], []
    for x in op.images(f):
        dx, dy = _grad(x)
        s = torch.sqrt(dx * dx + dy * dy + EPS * EPS)
        vals.append(s.sum())
        grads.append(_grad_t(dx / s, dy / s).reshape(-1))
    return torch.stack(vals), torch.cat(grads)


def exact(case, seed):
    call = case["call"]
    shaped = lambda x, *one: x if "uneven" in case else x.reshape(*([case["batch"]] if case["batch"] > 1 else []), *one)  # noqa: E731
    img = lambda x: shaped(x, case["n"], case["n"])  # noqa: E731
    dat = lambda x: shaped(x, case["n_det"], case["n_t"])  # noqa: E731
    if call == "pdhg_step":
        geoms, *v = _pdhg_start(case, seed)
        f, fbar, y, px, py, g = (x.double() for x in v)
        op, step = _Packed(geoms), math.sqrt(_solver_steps(geoms))
        sums, new, bars, pxs, pys = [], [], [], [], []
        y = (y + step * (op.forward(fbar) - g)) / (1 + step)
        at = op.adjoint(y)
        for x, xb, qx, qy, a in zip(*(op.images(z) for z in (f, fbar, px, py, at))):
            dx, dy = _grad(xb)
            qx, qy = qx + step * dx, qy + step * dy
            k = torch.clamp(LAM / torch.sqrt(qx * qx + qy * qy).clamp_min(1e-300), max=1.0)
            qx, qy = qx * k, qy * k
            nx = (x - step * (a + _grad_t(qx, qy))).clamp_min(0)
            sums += [((nx - x) ** 2).sum(), (nx ** 2).sum()]
            for to, z in zip((new, bars, pxs, pys), (nx, 2 * nx - x, qx, qy)):
                to.append(z.reshape(-1))
        return {"f": img(torch.cat(new)), "fbar": img(torch.cat(bars)), "y": dat(y), "px": img(torch.cat(pxs)),
                "py": img(torch.cat(pys)), "delta": torch.stack(sums)}
    geoms, f, g, _ = _inputs(case, seed)
    f, g, op = f.to(_dtype(case)).double(), g.double(), _Packed(geoms)
    if call == "forward":
        return dat(op.forward(f))
    if call == "adjoint":
        return img(op.adjoint(g))
    if call in ("pair", "graph_pair"):
        return dat(op.forward(f)), img(op.adjoint(g))
    if call == "tv_step":
        return img((f - _solver_steps(geoms) * (op.adjoint(op.forward(f) - g) + LAM * _tv(op, f)[1])).clamp_min(0))
    if call == "tv_grad":
        value, grad = _tv(op, f)
        return value, img(grad)
    if call == "tv_run":
        tau, f, changes = _solver_steps(geoms), torch.zeros_like(f), []
        for _ in range(case["iters"]):
            new = (f - tau * (op.adjoint(op.forward(f) - g) + LAM * _tv(op, f)[1])).clamp_min(0)
            changes.append(max(float(torch.linalg.norm(b - a) / torch.linalg.norm(b).clamp_min(1e-15))
                               for a, b in zip(op.images(f), op.images(new))))
            f = new
        return img(f), changes
    value, grad = _tv(op, f)
    r = op.forward(f) - g
    return (r * r).sum() + DIP_LAM * value.sum(), img(2 * op.adjoint(r) + DIP_LAM * grad)
