"""Neighbour lists that leave their row, and the viscous sum over them, against the oracle (needs a
GB300).  Sorted slots share the list blocks of their chunk.  Of every state it is checked, from brute
force lengths in the sorted order, that it is what it is named after: lists in a row and blocks, a
chunk that asks for more blocks than it has, or lists longer than all their blocks.

The bound of a viscous acceleration is the path's tolerance times the sum of the magnitudes that enter
it, each kernel taken at its centre and each velocity difference as the sum of both: rounding of the
kernel's argument, of the predicted velocities and of the sum are all within it.  The accelerations
themselves lie far above it, so that a sum left out or read from the wrong place does not pass."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

TOL = {32: 1e-5, 64: 1e-12}
CHUNK = 128
ROW, XB, NXB = {2: 32, 3: 128}, {2: 32, 3: 64}, {2: 128, 3: 128}   # the lists' shape
XMAX = 8


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def with_patches(w, patches, seed=3):
    """`w` with n more volume particles uniform in the ball (c, r) for every (c, r, n) of patches."""
    rng, xs = np.random.default_rng(seed), [w["x"]]
    D = w["domain"]["D"]
    for c, r, n in patches:
        d = rng.normal(size=(n, D))
        d *= (r * rng.random((n, 1)) ** (1 / D)) / np.linalg.norm(d, axis=1, keepdims=True)
        x = np.zeros((n, 3))
        x[:, :D] = np.asarray(c)[:D] + d
        xs.append(x)
    x = np.concatenate(xs)
    return dict(w, x=x, group=np.concatenate([w["group"], np.zeros(len(x) - len(w["x"]), np.int32)]))


def graded_ball():
    """A ball with coarse particles at its centre beside finer ones, thinned outside |x| < 0.4."""
    w = WL.sphere02(mc_samples=100_000)
    r = np.linalg.norm(w["x"], axis=1)
    return WL.subset(w, (r < 0.4) | (np.arange(len(r)) % 4 == 0))


def state(name):
    if name.startswith("square"):
        w = WL.square2d(h=0.02, seed=2)
        spots = [(0.25, 0.2), (0.7, 0.45), (0.4, 0.7)]
        return with_patches(w, {"square_blocks": [(c, 0.02, 45) for c in spots],
                                "square_out_of_blocks": [((0.5, 0.5), 0.12, 900)],
                                "square_longer_than_blocks": [((0.5, 0.5), 0.02, 400)]}[name])
    return with_patches(graded_ball(), {"ball_blocks": [], "ball_out_of_blocks": [((0, 0, 0), 0.3, 350)],
                                        "ball_longer_than_blocks": [((0, 0, 0), 0.3, 2000)]}[name])


def neighbours(w, h, i):
    """Indices and distances within the larger of the pair's and the particle's own support."""
    r = np.linalg.norm(w["x"] - w["x"][i], axis=1)
    k = w["params"]["kappa"]
    j = np.flatnonzero(r < k * np.maximum(h[i], 0.5 * (h[i] + h)))
    return j, r[j]


def viscous_scale(w, h, vt, dim, i):
    j, r = neighbours(w, h, i)
    p, d, g = w["params"], dim[i], w["group"]
    R = 0.5 * p["kappa"] * (h[i] + h[j])
    keep = (g[j] == g[i]) & (j != i) & (r < R)
    j, R = j[keep], R[keep]
    speed = np.linalg.norm(vt, axis=1)
    eta = p["visc"] * p["kappa"] * h ** (1.0 - d) * speed
    eb = 2 * eta[i] * eta[j] / np.maximum(eta[i] + eta[j], 1e-300)
    alpha = {1: 1.5 / R, 2: 7 / math.pi / R ** 2, 3: 10.5 / math.pi / R ** 3}[d]
    return float((eb * (h[i] ** (2 * d) + h[j] ** (2 * d)) * 20 * alpha / R ** 2 * (speed[i] + speed[j])).sum())


@pytest.mark.parametrize("name,prec", [(f"{s}_{k}", p) for s in ("square", "ball") for p in (32, 64)
                                       for k in ("blocks", "out_of_blocks", "longer_than_blocks")])
def test_pair_sums_over_long_lists(name, prec):
    w = state(name)
    D, n = w["domain"]["D"], len(w["x"])
    t = np.float32 if prec == 32 else np.float64
    h = O.Oracle(w).h.astype(t).astype(np.float64)
    v = np.zeros((n, 3))
    v[:, :D] = np.random.default_rng(5).normal(0, 2e-3, (n, D)).astype(t)
    m = S.Mesh(w, precision=prec)
    m.set_state(v=v, h=h)
    # the state is what its name says
    _, _, perm = S.sph_debug_rebuild(m.h, n, S.sph_mesh_grid(m.h).n_cells)
    length = np.array([len(neighbours(w, h, i)[0]) for i in range(n)])
    need = np.minimum(np.maximum(-((ROW[D] - length[perm]) // XB[D]), 0), XMAX)
    asked = np.add.reduceat(need, np.arange(0, n, CHUNK))
    most = ROW[D] + XMAX * XB[D]
    kind = name.split("_", 1)[1]
    assert length.max() > ROW[D] + (XB[D] if kind == "blocks" else 0)
    assert (asked.max() > 1.1 * NXB[D]) == (kind != "blocks") and (kind != "blocks" or asked.max() < 0.9 * NXB[D])
    assert (length.max() > 1.1 * most) == (kind == "longer_than_blocks")
    long = np.argsort(length)[-300:]
    sub = np.unique(np.concatenate([long, np.random.default_rng(2).choice(n, 200, replace=False)]))
    tol = TOL[prec]
    o = O.Oracle(w, h=h, v=v)
    ref = o.interact(sub=sub)
    got = S.sph_debug_interact(m.h, n, m.n_groups)
    err = np.linalg.norm(got["a_p"][sub] - ref["a_p"], axis=1)
    assert np.all(err <= tol * ref["S"] + 1e-300), (err / np.maximum(ref["S"], 1e-300)).max()
    moving = o.gdim[w["group"][sub]] > 0
    for key in ("sigma", "gamma"):
        assert np.allclose(got[key][sub][moving], ref[key][moving], rtol=10 * tol, atol=0)
    # the viscous sum from the device's own a_p, with the step size of Eq. 24
    dt, eps, f = np.where(o.gdim > 0, np.minimum(got["dta"], 1e3), 0.0), 0.1, 0.75
    dt = dt.astype(t).astype(np.float64)
    o.set_step_params(dt, [0] * o.G, eps, f)
    av = o.integrate(got["a_p"], sub=sub)["a_v"]
    out = S.sph_debug_update(m.h, n, dt, np.zeros(o.G, np.int32), eps, f)
    vt = f * v + dt[w["group"]][:, None] * (got["a_p"] - eps * f * v)
    dim = o.gdim[w["group"]]
    bound = np.array([tol * viscous_scale(w, h, vt, dim, i) if dim[i] > 0 else 1e-300 for i in sub])
    err = np.linalg.norm(out["a_v"][sub] - av, axis=1)
    assert np.all(err <= bound), (err / bound).max()
    size = np.linalg.norm(av, axis=1) / bound
    assert np.median(size[moving]) > 30 and np.median(size[np.isin(sub, long) & moving]) > 30, size
    m.close()


# 16 particles per warp in 3D, with a ragged last chunk
def test_neighbor_sets_of_a_large_cube():
    n = 524_291
    w = WL.cube_sphere(n_target=n + 3000, seed=2, mc_samples=100_000)
    w = WL.subset(w, np.sort(np.random.default_rng(11).permutation(len(w["x"]))[:n]))
    h = O.Oracle(w).h.astype(np.float32).astype(np.float64)
    m = S.Mesh(w, precision=32)
    m.set_state(h=h)
    counts, lists = S.sph_debug_neighbors(m.h, n, 0)
    off = np.concatenate([[0], np.cumsum(counts)])
    g = S.sph_mesh_grid(m.h)
    og = O.grid_spec(3, w["domain"]["lo"], w["domain"]["hi"], w["h_lo"], w["h_hi"], kappa=w["params"]["kappa"],
                     cells_per_support=g.cells_per_support)
    for i in np.concatenate([np.random.default_rng(1).choice(n, 30, replace=False), np.arange(n - 3, n)]):
        ref = O.neighbors_repr(og, w["x"], h, int(i), prec=32, kappa=w["params"]["kappa"])
        assert np.array_equal(lists[off[i]:off[i + 1]], ref), i
    m.close()


# one update kernel up to 65,536 slots in 2D, three above
@pytest.mark.parametrize("n", [65_400, 65_700])
def test_update_at_the_2d_kernel_split(n):
    w = WL.disk_holes(n_target=n + 1500, seed=4, mc_samples=100_000)
    w = WL.subset(w, np.sort(np.random.default_rng(11).permutation(len(w["x"]))[:n]))
    h = O.Oracle(w).h.astype(np.float32).astype(np.float64)
    v = np.zeros((n, 3))
    v[:, :2] = np.random.default_rng(5).normal(0, 2e-3, (n, 2)).astype(np.float32)
    o = O.Oracle(w, h=h, v=v)
    r = o.interact()
    dt = np.where(o.gdim > 0, np.minimum(r["dta"], 1e3), 0.0)
    o.set_step_params(dt, [0] * o.G, 0.1, 0.75)
    ref = o.integrate(r["a_p"])
    m = S.Mesh(w, precision=32)
    m.set_state(h=h, v=v)
    got = S.sph_debug_update(m.h, n, dt, np.zeros(o.G, np.int32), 0.1, 0.75)
    vs = dt[w["group"]] * r["S"] + np.linalg.norm(v, axis=1) + 1e-300
    moving = o.gdim[w["group"]] > 0
    ev = np.linalg.norm(got["v"] - ref["v"], axis=1)
    assert np.all(ev[moving] <= 50 * TOL[32] * vs[moving]), (ev / vs)[moving].max()
    m.close()
