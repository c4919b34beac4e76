"""What a user of the library has it do, as measured cases.

A pass of most cases is what a meshing program does between two looks at its particles: ten
relaxation steps and the particles read back.  Around it stand a whole job from host arrays,
a batch of independent problems in one handle, and a server that draws and relaxes a queue of
jobs.  `exact` relaxes the same particles in 64 bits with plain torch (Algorithm 1 with the
sums of Eqs. 7, 18-20, the step sizes of Eq. 24 and the projections).

Initial particles are drawn here from the seed, with probability proportional to the target
density h^-d (volume, surfaces) or spaced by it (curves), as the method starts from.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

STEPS = 10          # relaxation steps between two looks at the particles
SERVE_STEPS = 20    # iterations of a served job (one scheduling round of the server)
DEV = "cuda" if torch.cuda.is_available() else "cpu"
EXACT_MOST = 400_000   # particles beyond which `exact` would take over about 20 seconds


def listed():
    return [
        # the smallest 2D mesh of the tests and examples: one step is a chain of short kernels,
        # its time is latency and launches
        dict(name="square_2601", call="relax", shape="square", n=2601, precision=32, order=0),
        # the Square of the method's own comparison, in the 64-bit build that a user takes for
        # reference runs
        dict(name="paper_square_f64", call="relax", shape="square_radial", n=2915, precision=64, order=0),
        # an ordinary 2D mesh with curved boundaries and graded spacing
        dict(name="disk_20k", call="relax", shape="disk", n=20_000, precision=32, order=0),
        # the 2D benchmark workload
        dict(name="disk_120k", call="relax", shape="disk", n=120_000, precision=32, order=0),
        # the largest 2D mesh
        dict(name="disk_1m", call="relax", shape="disk", n=1_000_000, precision=32, order=0),
        # a small 3D case of the method's tables, with its feature loop taken in sequence (three
        # re-sorted passes per step)
        dict(name="sphere02_order", call="relax", shape="sphere02", n=26_514, precision=32, order=1),
        # the Cube of the method's tables: an ordinary 3D mesh with strongly graded spacing
        dict(name="paper_cube_83k", call="relax", shape="cube_radial", n=82_922, precision=32, order=0),
        # a whole job from host arrays: load, relax, read back
        dict(name="cube_300k_job", call="job", shape="cube", n=300_000, precision=32, order=0),
        # the headline workload, the largest 3D mesh
        dict(name="cube_1.2m", call="relax", shape="cube", n=1_200_000, precision=32, order=0),
        # a 3D mesh in 64 bits, of the size of the jobs served one at a time
        dict(name="cube_40k_f64", call="relax", shape="cube", n=40_000, precision=64, order=0),
        # twelve independent 3D problems of 1k to 100k particles stepped together
        dict(name="batch_3d_12", call="batch", shape="cube", n=100_000, instances=12, precision=32, order=0),
        # a queue of eight jobs, 2D and 3D, given by their problems alone and drawn on the device
        dict(name="serve_8", call="serve", shape="mix", n=60_000, instances=8, precision=32, order=0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["relax"] * 5 + ["job", "batch", "serve"])
    if call == "serve":
        return dict(call=call, shape="mix", n=_log_uniform(rng, 2_000, 60_000), instances=rng.randint(2, 8), precision=32, order=0)
    shape = rng.choice(["disk", "cube"])
    if call == "batch":
        return dict(call=call, shape=shape, n=_log_uniform(rng, 2_000, 100_000), instances=rng.randint(2, 12), precision=32, order=0)
    kind = rng.choice(["plain", "plain", "plain", "f64", "order"])
    top = {"plain": 1_000_000, "f64": 40_000, "order": 60_000}[kind]
    return dict(call=call, shape=shape, n=_log_uniform(rng, 1_000, top), precision=64 if kind == "f64" else 32,
                order=1 if kind == "order" else 0)


# ------------------------------------------------------------------------------------------
# problems and their initial particles
# ------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _problem(shape, n, geometry_seed):
    """Domain, sizing, parameters and particles per feature (no particles)."""
    if shape in ("square_radial", "cube_radial", "sphere02"):
        w = getattr(WL, shape)(mc_samples=100_000)
        return dict(w, counts=np.bincount(w["group"], minlength=len(w["domain"]["features"])).tolist())
    build = WL.disk_holes if shape == "disk" else WL.cube_sphere
    w = build(n_target=n, seed=geometry_seed, mc_samples=100_000, sample=False)
    counts = [_count(f, w["domain"], w["sizing"]) for f in w["domain"]["features"]]
    return dict(w, counts=counts)


def _sizing(z, x):
    if z["kind"] == "const":
        return torch.full_like(x[:, 0], z["a"])
    if z["kind"] == "radial":
        d = (x - x.new_tensor(z["q"])).norm(dim=1)
    else:
        d = torch.full_like(x[:, 0], math.inf)
        for c, r in z["refs"]:
            d = torch.minimum(d, ((x - x.new_tensor(c)).norm(dim=1) - r).abs())
    return (z["a"] + z["b"] * d).clamp(z["lo"], z["hi"])


def _phi(dom, x):
    """Level set of the domain (positive inside) and its gradient."""
    phi, grad = torch.full_like(x[:, 0], math.inf), torch.zeros_like(x)

    def lower(p, g):
        nonlocal phi, grad
        phi, grad = torch.minimum(phi, p), torch.where((p < phi)[:, None], g, grad)

    if dom["base"] == "box":
        for a in range(dom["D"]):
            e = torch.zeros_like(x)
            e[:, a] = 1.0
            lower(x[:, a] - dom["lo"][a], e)
            lower(dom["hi"][a] - x[:, a], -e)
    else:
        d = x - x.new_tensor(dom["ball_c"])
        r = d.norm(dim=1)
        lower(dom["ball_r"] - r, -d / r.clamp_min(1e-300)[:, None])
    for c, hr in dom["holes"]:
        d = x - x.new_tensor(c)
        r = d.norm(dim=1)
        lower(r - hr, d / r.clamp_min(1e-300)[:, None])
    return phi, grad


def _uniform(f, dom, m, gen):
    """m points uniform on a surface or in the volume's bounding box, and the measure they cover."""
    u = lambda k: torch.rand(m, k, generator=gen, device=DEV, dtype=torch.float64)  # noqa: E731
    at = lambda v: torch.tensor(v, device=DEV, dtype=torch.float64)  # noqa: E731
    if f["kind"] == "volume":
        D, lo, hi = dom["D"], at(dom["lo"]), at(dom["hi"])
        x = torch.zeros(m, 3, device=DEV, dtype=torch.float64)
        x[:, :D] = lo[:D] + u(D) * (hi - lo)[:D]
        return x, float((hi - lo)[:D].prod())
    if f["kind"] == "rect":
        st = u(2) * at([f["lu"], f["lw"]])
        return at(f["o"]) + st[:, :1] * at(f["u"]) + st[:, 1:] * at(f["w"]), f["lu"] * f["lw"]
    g = torch.randn(m, 3, generator=gen, device=DEV, dtype=torch.float64)
    return at(f["c"]) + f["r"] * g / g.norm(dim=1, keepdim=True), 4 * math.pi * f["r"] ** 2


def _accept(f, dom, z, x, gen):
    """Rejection with probability (h_min/h)^d, off the boundary by a quarter of h."""
    h = _sizing(z, x)
    keep = torch.rand(len(x), generator=gen, device=DEV, dtype=torch.float64) < (z["lo"] / h) ** f["dim"]
    if f["kind"] == "volume":
        keep &= _phi(dom, x)[0] > 0.25 * h
    elif f["kind"] == "rect":
        for e, L in (("u", f["lu"]), ("w", f["lw"])):
            s = ((x - x.new_tensor(f["o"])) * x.new_tensor(f[e])).sum(1)
            keep &= (s > 0.25 * h) & (s < L - 0.25 * h)
    return keep


def _curve(f, s):
    """Points at the fractions s of a curve, and its length."""
    if f["kind"] == "segment":
        a, b = np.asarray(f["a"], float), np.asarray(f["b"], float)
        return a + s[:, None] * (b - a), float(np.linalg.norm(b - a))
    t = 2 * math.pi * s
    return np.asarray(f["c"], float) + f["r"] * np.stack([np.cos(t), np.sin(t), 0 * t], 1), 2 * math.pi * f["r"]


def _line_density(f, z):
    s = (np.arange(4096) + 0.5) / 4096
    x, length = _curve(f, s)
    return 1.0 / _sizing(z, torch.from_numpy(x)).numpy(), length


def _count(f, dom, z):
    """Particles of a feature: the integral of h^-d over it."""
    if f["dim"] == 0:
        return 1
    if f["dim"] == 1:
        rho, length = _line_density(f, z)
        return int(round(float(rho.mean()) * length))
    gen = torch.Generator(DEV).manual_seed(1)
    x, measure = _uniform(f, dom, 2_000_000 if f["kind"] == "volume" else 200_000, gen)
    rho = _sizing(z, x) ** -float(f["dim"])
    if f["kind"] == "volume":
        rho = rho * (_phi(dom, x)[0] > 0)
    return int(round(float(rho.mean()) * measure))


def _particles(w, seed):
    """(x [n][3] float64, group [n] int32) on the host."""
    gen, rng = torch.Generator(DEV).manual_seed(seed), np.random.default_rng(seed)
    dom, z, xs, gs = w["domain"], w["sizing"], [], []
    for k, (f, n) in enumerate(zip(dom["features"], w["counts"])):
        if f["dim"] == 0:
            x = np.asarray([f["p"]], float)
        elif f["dim"] == 1:
            rho, _ = _line_density(f, z)
            cdf = np.concatenate([[0.0], np.cumsum(rho)]) / rho.sum()
            closed = f["kind"] == "circle"
            u = (np.arange(n) + rng.uniform(-0.1, 0.1, n) + (0 if closed else 1)) / (n if closed else n + 1)
            x = _curve(f, np.interp(np.mod(u, 1.0), cdf, np.linspace(0.0, 1.0, 4097)))[0]
        else:
            got, have = [], 0
            while have < n:
                c, _ = _uniform(f, dom, min(max(16 * (n - have), 1 << 14), 1 << 23), gen)
                got.append(c[_accept(f, dom, z, c, gen)])
                have += len(got[-1])
            x = torch.cat(got)[:n].cpu().numpy()
        xs.append(x)
        gs.append(np.full(len(x), k, np.int32))
    return np.concatenate(xs), np.concatenate(gs)


def _sizes(case):
    """Particle targets of a batch's or a queue's problems: spread over [1k, n] by their logarithm."""
    k = case["instances"]
    return [int(round(1000 * (case["n"] / 1000) ** (i / max(k - 1, 1)))) for i in range(k)]


def _workloads(case, seed):
    """The problems of a case with their particles."""
    if case["shape"] == "square":
        ws = [WL.square2d(h=1.0 / round(math.sqrt(case["n"]) - 1), seed=seed)]
    elif case["call"] == "serve":
        # 2D and 3D in turn; the server draws the particles
        ws = [_problem("disk" if i % 2 == 0 else "cube", n, 20 + i) for i, n in enumerate(_sizes(case))]
    else:
        sizes = _sizes(case) if case["call"] == "batch" else [case["n"]]
        ws = [_problem(case["shape"], n, 2 + i) for i, n in enumerate(sizes)]
        xg = [_particles(w, seed * 100 + i) for i, w in enumerate(ws)]
        ws = [dict(w, x=x, group=g) for w, (x, g) in zip(ws, xg)]
    more = dict(group_convergence=1, feature_order=1) if case["order"] else {}
    return [dict(w, params=dict(w["params"], **more)) for w in ws]


# ------------------------------------------------------------------------------------------
# the measured calls
# ------------------------------------------------------------------------------------------
def prepare(case, seed):
    ws = _workloads(case, seed)
    state = dict(case=case, seed=seed, ws=ws)
    if case["call"] == "serve":
        state["server"] = S.Server(precision=case["precision"], max_jobs=case["instances"])
    elif case["call"] == "batch":
        b = S.Batch(ws, precision=case["precision"])
        for i, w in enumerate(ws):
            b.set_state(i, w["x"], w["group"])
        state["batch"] = b
    else:
        m = S.Mesh(ws[0], precision=case["precision"])
        if case["call"] == "relax":
            m.set_state()
        state["mesh"] = m
    return state


def _out(p, precision):
    """The particles in the precision that the handle works in (its v and h are such values)."""
    t = np.float32 if precision == 32 else np.float64
    return {k: a if k == "group" else a.astype(t) for k, a in p.items()}


def run(state):
    case, prec = state["case"], state["case"]["precision"]
    if case["call"] == "serve":
        server = state["server"]
        ids = [server.submit_sampled(w, SERVE_STEPS, state["seed"] * 100 + i) for i, w in enumerate(state["ws"])]
        server.drain()
        out = []
        for j in ids:
            info, p = server.job(j)
            out.append(dict(_out(p, prec), iterations=int(info.iterations)))
            server.release(j)
        return out
    if case["call"] == "batch":
        b = state["batch"]
        b.step(STEPS)
        return [_out(b.positions(i), prec) for i in range(b.n_inst)]
    m = state["mesh"]
    if case["call"] == "job":
        m.set_state()
    m.step(STEPS)
    return _out(m.positions(), prec)


def work(case):
    """Per step each particle's state (cell, offset, velocity, h, feature, index) read and written,
    50 operations per interacting pair in the pressure sum and 20 in the viscous one; then the
    particles handed over once."""
    word = case["precision"] // 8
    sizes = _sizes(case) if "instances" in case else [case["n"]]
    dims = [2 if case["shape"] in ("square", "square_radial", "disk") else 3] * len(sizes)
    if case["call"] == "serve":
        dims = [2 + i % 2 for i in range(len(sizes))]
    steps = SERVE_STEPS if case["call"] == "serve" else STEPS
    pairs = {2: math.pi * 2.6 ** 2, 3: 4 / 3 * math.pi * 2.6 ** 3}
    nbytes = flops = 0.0
    for n, D in zip(sizes, dims):
        nbytes += n * (steps * 2 * (D * (4 + 2 * word) + word + 8) + 60)
        if case["call"] == "job":
            nbytes += n * 28
        flops += n * steps * 70 * pairs[D]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------
# the same relaxation in 64 bits
# ------------------------------------------------------------------------------------------
def _morton(x):
    q = ((x - x.amin(0)) / (x.amax(0) - x.amin(0)).amax() * 1023).long()
    code = torch.zeros_like(q[:, 0])
    for b in range(10):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return code.argsort()


def _pairs(x, h, kappa):
    """Index pairs i != j with r < kappa max(h_i, (h_i + h_j)/2), by blocks of nearby particles."""
    order, out = _morton(x), []
    for i in order.split(256):
        gap = (x[i].amin(0) - x).clamp_min(0) + (x - x[i].amax(0)).clamp_min(0)
        hi = h[i].max()
        j = (gap.square().sum(1) < (kappa * torch.maximum(hi, 0.5 * (hi + h))).square()).nonzero()[:, 0]
        r2 = sum((x[i][:, a, None] - x[j][None, :, a]).square() for a in range(3))
        R = kappa * torch.maximum(h[i][:, None].expand_as(r2), 0.5 * (h[i][:, None] + h[j][None, :]))
        a, b = (r2 < R * R).nonzero(as_tuple=True)
        a, b = i[a], j[b]
        out.append(torch.stack([a[a != b], b[a != b]]))
    return torch.cat(out, 1)


def _kernel(d, r, R):
    """Wendland C2 of support R in d dimensions: W and dW/dr."""
    alpha = torch.where(d == 1, 1.5 / R, torch.where(d == 2, 7 / math.pi / R ** 2, 21 / (2 * math.pi) / R ** 3))
    q = (r / R).clamp_max(1.0)
    return alpha * (1 - q) ** 4 * (1 + 4 * q), alpha * -20 * q * (1 - q) ** 3 / R


class _Relaxation:
    def __init__(self, w):
        t = lambda v: torch.as_tensor(np.asarray(v), device=DEV)  # noqa: E731
        self.w, self.p, self.dom = w, w["params"], w["domain"]
        self.feats = self.dom["features"]
        self.x, self.group = t(w["x"]), t(w["group"]).long()
        self.dim = t([f["dim"] for f in self.feats])[self.group].double()
        self.v = torch.zeros_like(self.x)
        self.h = _sizing(w["sizing"], self.x)
        self.n, self.before = 0, {}

    def members(self):
        for g, f in enumerate(self.feats):
            at = (self.group == g).nonzero()[:, 0]
            if len(at):
                yield g, f, at

    def tangents(self):
        """Unit tangent of curve particles, unit normal of surface particles."""
        t = torch.zeros_like(self.x)
        for _, f, at in self.members():
            if f["kind"] == "segment":
                e = self.x.new_tensor(f["b"]) - self.x.new_tensor(f["a"])
                t[at] = e / e.norm()
            elif f["kind"] == "rect":
                t[at] = self.x.new_tensor(f["nb"])
            elif f["kind"] in ("circle", "sphere"):
                d = self.x[at] - self.x.new_tensor(f["c"])
                d = d / d.norm(dim=1, keepdim=True)
                t[at] = torch.stack([-d[:, 1], d[:, 0], 0 * d[:, 0]], 1) if f["kind"] == "circle" else d
        return t

    def normals(self):
        """Outward normal of every particle on a boundary feature."""
        nb = torch.zeros_like(self.x)
        for _, f, at in self.members():
            if f["kind"] in ("circle", "sphere"):
                d = self.x[at] - self.x.new_tensor(f["c"])
                nb[at] = f["orient"] * d / d.norm(dim=1, keepdim=True)
            elif f["kind"] != "volume":
                nb[at] = self.x.new_tensor(f["nb"])
        return nb

    def onto(self, t, dim, a):
        s = (a * t).sum(1, keepdim=True)
        d = dim[:, None]
        return torch.where(d == self.dom["D"], a, torch.where(d == 0, 0 * a, torch.where(d == 1, s * t, a - s * t)))

    def project(self, f, x):
        at = x.new_tensor
        if f["kind"] == "segment":
            e = at(f["b"]) - at(f["a"])
            s = (((x - at(f["a"])) * e).sum(1) / (e * e).sum()).clamp(0, 1)
            return at(f["a"]) + s[:, None] * e
        if f["kind"] == "rect":
            s = ((x - at(f["o"])) * at(f["u"])).sum(1).clamp(0, f["lu"])
            t = ((x - at(f["o"])) * at(f["w"])).sum(1).clamp(0, f["lw"])
            return at(f["o"]) + s[:, None] * at(f["u"]) + t[:, None] * at(f["w"])
        d = x - at(f["c"])
        return at(f["c"]) + f["r"] * d / d.norm(dim=1, keepdim=True)

    def one_pass(self, moves):
        """One pass over the particles of `moves`: forces, step sizes, update, projection."""
        p, x, h, dim, group = self.p, self.x, self.h, self.dim, self.group
        kappa, D, N = p["kappa"], self.dom["D"], len(x)
        i, j = _pairs(x, h, kappa)
        keep = moves[i]
        i, j = i[keep], j[keep]
        dx = x[i] - x[j]
        r = dx.norm(dim=1)
        R, d = 0.5 * kappa * (h[i] + h[j]), dim[i]
        same, near = group[i] == group[j], r < 0.5 * kappa * (h[i] + h[j])
        one = torch.ones_like(h)
        # Eqs. 20, 18
        W, _ = _kernel(d, r, kappa * h[i])
        W = W * (same & (r < kappa * h[i]))
        W0, _ = _kernel(dim.clamp_min(1), 0 * h, kappa * h)
        gam = (W0 * h ** dim).index_add(0, i, W * h[j] ** d)
        # Eq. 19
        Wij, dW = _kernel(d, r, R)
        P = p["p0"] * (h[i] ** (2 * d) + h[j] ** (2 * d))
        pair = same & near & (r > 0)
        F = torch.zeros_like(x).index_add(0, i, (P * dW / r.clamp_min(1e-300) * pair)[:, None] * dx)
        t, nb = self.tangents(), self.normals()
        wall = ((dim[j] < d) & near).nonzero()[:, 0]
        n = self.onto(t[i[wall]], d[wall], nb[j[wall]])
        n2 = (n * n).sum(1)
        c = P[wall] * Wij[wall] / h[j[wall]] * (n2 > 1e-12) / n2.clamp_min(1e-12).sqrt()
        F = F.index_add(0, i[wall], c[:, None] * n)
        ap = self.onto(t, dim, -F / gam[:, None]) * moves[:, None]
        # Eq. 24, per feature
        dt, rs = 0 * one, torch.ones_like(moves)
        for g, f, at in self.members():
            if f["dim"] == 0 or not bool(moves[at[0]]):
                continue
            a, v, rc = ap[at].norm(dim=1), self.v[at].norm(dim=1), kappa * h[at]
            dta = float(torch.where(a > 0, p["cfl_a"] * (rc / a).sqrt(), torch.inf).min())
            dtv = float(torch.where(v > 0, p["cfl_v"] * rc / v, torch.inf).min())
            old, cand = self.before.get(g, 0.0), min(dta, dtv)
            still = self.n % p["reset_period"] == 0 or (old > 0 and cand < p["dt_collapse"] * old)
            self.before[g] = min(dta if still else cand, p["dt_cap"])
            dt[at], rs[at] = self.before[g], still
        # Eqs. 23, 7, 8
        v = torch.where(rs[:, None], 0 * self.v, self.v)
        vt = v + dt[:, None] * (ap - p["eps1"] * v)
        eta = p["visc"] * kappa * h * vt.norm(dim=1) / h ** dim
        both = eta[i] + eta[j]
        eb = torch.where(both > 0, 2 * eta[i] * eta[j] / both.clamp_min(1e-300), 0 * both)
        c = eb * (h[i] ** (2 * d) + h[j] ** (2 * d)) * dW / r.clamp_min(1e-300) * pair
        av = self.onto(t, dim, torch.zeros_like(x).index_add(0, i, c[:, None] * (vt[i] - vt[j])))
        vn = vt + dt[:, None] * av
        xn = x + dt[:, None] * vn
        for _, f, at in self.members():
            if f["dim"] == 0 or not bool(moves[at[0]]):
                continue
            if f["kind"] != "volume":
                xn[at] = self.project(f, xn[at])
                continue
            y, vy, target = xn[at], vn[at], 0.01 * h[at]
            phi, grad = _phi(self.dom, y)
            out = phi < 0
            for _ in range(3):
                back = out & (phi < 0.5 * target)
                y = torch.where(back[:, None], y + ((target - phi) / (grad * grad).sum(1))[:, None] * grad, y)
                phi, grad = _phi(self.dom, y)
            xn[at], vn[at] = y, torch.where(out[:, None], 0 * vy, vy)
        self.x = torch.where(moves[:, None], xn, x)
        t = self.tangents()
        vn = torch.where((dim < D)[:, None], self.onto(t, dim, vn), vn)
        self.v = torch.where(moves[:, None], vn, self.v)
        self.h = torch.where(moves, _sizing(self.w["sizing"], self.x), h)

    def step(self):
        if self.p.get("feature_order"):
            for c in range(1, self.dom["D"] + 1):
                self.one_pass(self.dim == c)
        else:
            self.one_pass(self.dim > 0)
        self.n += 1


def exact(case, seed):
    if case["call"] == "serve":
        return None   # its particles are the library's own drawing
    ws = _workloads(case, seed)
    if sum(len(w["x"]) for w in ws) > EXACT_MOST:
        return None
    out = []
    for w in ws:
        s = _Relaxation(w)
        for _ in range(STEPS):
            s.step()
        out.append(dict(x=s.x.cpu().numpy(), v=s.v.cpu().numpy(), h=s.h.cpu().numpy(), group=None))
    return out if case["call"] == "batch" else out[0]
