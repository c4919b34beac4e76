"""The neighbour search and its lists at the edges of their ranges, against the oracle (needs a GB300).

* every width of the search (2, 4, 8 or 16 particles per warp, by the slots of the batch): the
  neighbour sets of sampled particles, and of all particles next to the ragged end, equal brute
  force on the stored representation;
* lists longer than a row (blocks), lists of a chunk that runs out of blocks, and overflowed lists:
  a_p, sigma and gamma of the pressure pass, and the update, within the path's bounds;
* the update as one kernel and as three, on both sides of the sizes where the path changes.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

TOL = {32: 1e-5, 64: 1e-12}


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def float32_h(w):
    return O.Oracle(w).h.astype(np.float32).astype(np.float64)


def first(w, n):
    """The first n particles in a seeded random order (a ragged last chunk and a ragged last warp)."""
    keep = np.sort(np.random.default_rng(11).permutation(len(w["x"]))[:n])
    return WL.subset(w, keep)


# slots just below and above the sizes at which the width changes, with ragged last warps
@pytest.mark.parametrize("shape,n", [("disk", 3001), ("disk", 65_409), ("disk", 65_537), ("disk", 524_291),
                                     ("cube", 8_193), ("cube", 32_769), ("cube", 65_537)])
def test_neighbor_sets_at_every_search_width(shape, n):
    make = WL.disk_holes if shape == "disk" else WL.cube_sphere
    w = first(make(n_target=n + n // 50, seed=2, mc_samples=100_000), n)
    h = float32_h(w)
    m = S.Mesh(w, precision=32)
    m.set_state(h=h)
    counts, lists = S.sph_debug_neighbors(m.h, m.n, 0)
    off = np.concatenate([[0], np.cumsum(counts)])
    g = S.sph_mesh_grid(m.h)
    og = O.grid_spec(w["domain"]["D"], w["domain"]["lo"], w["domain"]["hi"], w["h_lo"], w["h_hi"],
                     kappa=w["params"]["kappa"], cells_per_support=g.cells_per_support)
    idx = np.random.default_rng(1).choice(n, 40, replace=False)
    for i in np.concatenate([idx, np.arange(n - 3, n)]):
        ref = O.neighbors_repr(og, w["x"], h, int(i), prec=32, kappa=w["params"]["kappa"])
        assert np.array_equal(lists[off[i]:off[i + 1]], ref), i
    m.close()


def graded_ball(extra):
    """Sphere02 (coarse particles at the centre beside finer ones around), thinned outside |x| < 0.4,
    with `extra` more particles close to the centre."""
    w = WL.sphere02(mc_samples=100_000)
    r = np.linalg.norm(w["x"], axis=1)
    w = WL.subset(w, (r < 0.4) | (np.arange(len(r)) % 4 == 0))
    rng = np.random.default_rng(3)
    x = rng.normal(size=(extra, 3))
    x *= (0.3 * rng.random((extra, 1)) ** (1 / 3)) / np.linalg.norm(x, axis=1, keepdims=True)
    return dict(w, x=np.concatenate([w["x"], x]), group=np.concatenate([w["group"], np.zeros(extra, np.int32)]))


# extra = 0: lists of up to about 260 candidates in a row and blocks; 350: lists that fit the blocks,
# in chunks that run out of them; 2,000: lists longer than all their blocks
@pytest.mark.parametrize("extra,prec,longest", [(0, 32, 128), (0, 64, 128), (350, 32, 400), (2_000, 32, 640)])
def test_long_lists(extra, prec, longest):
    w = graded_ball(extra)
    h = O.Oracle(w).h if prec == 64 else float32_h(w)
    m = S.Mesh(w, precision=prec)
    m.set_state(h=h)
    counts, _ = S.sph_debug_neighbors(m.h, m.n, 1)
    assert counts.max() > longest
    sub = np.unique(np.concatenate([np.argsort(counts)[-300:], np.random.default_rng(2).choice(m.n, 300, replace=False)]))
    o = O.Oracle(w, h=h)
    got = S.sph_debug_interact(m.h, m.n, m.n_groups)
    ref = o.interact(sub=sub, use_grid=True)
    tol = TOL[prec]
    err = np.linalg.norm(got["a_p"][sub] - ref["a_p"], axis=1)
    assert np.all(err <= tol * ref["S"] + 1e-300), (err / np.maximum(ref["S"], 1e-300)).max()
    for key in ("sigma", "gamma"):
        assert np.allclose(got[key][sub], ref[key], rtol=10 * tol, atol=0)
    # the viscous pass over the same lists: the oracle's update from the GPU's own a_p
    dt = np.where(o.gdim > 0, 1e-3, 0.0)
    o.set_step_params(dt, [1] * o.G, 0.0, 1.0)
    upd = o.integrate(got["a_p"], use_grid=True)
    out = S.sph_debug_update(m.h, m.n, dt, np.ones(o.G, np.int32), 0.0, 1.0)
    scale = np.abs(upd["v"]).max()
    assert np.abs(out["v"] - upd["v"]).max() <= 50 * tol * scale
    m.close()


# one kernel up to 32,768 slots in 2D and 8,192 in 3D (FP32), three above and in the FP64 build
@pytest.mark.parametrize("shape,n,prec", [("disk", 32_700, 32), ("disk", 33_000, 32), ("cube", 8_100, 32),
                                          ("cube", 8_300, 32), ("disk", 2_000, 64)])
def test_update_on_both_sides_of_the_kernel_split(shape, n, prec):
    make = WL.disk_holes if shape == "disk" else WL.cube_sphere
    w = first(make(n_target=n + n // 20, seed=4, mc_samples=100_000), n)
    D = w["domain"]["D"]
    h = O.Oracle(w).h if prec == 64 else float32_h(w)
    v = np.zeros((n, 3))
    v[:, :D] = np.random.default_rng(5).normal(0, 2e-3, (n, D)).astype(np.float32)
    o = O.Oracle(w, h=h, v=v)
    r = o.interact(use_grid=True)
    dt = np.where(o.gdim > 0, np.minimum(r["dta"], 1e3), 0.0)
    o.set_step_params(dt, [0] * o.G, 0.1, 0.75)
    ref = o.integrate(r["a_p"], use_grid=True)
    m = S.Mesh(w, precision=prec)
    m.set_state(h=h, v=v)
    got = S.sph_debug_update(m.h, m.n, dt, np.zeros(o.G, np.int32), 0.1, 0.75)
    vs = dt[w["group"]] * r["S"] + np.linalg.norm(v, axis=1) + 1e-300
    moving = o.gdim[w["group"]] > 0
    ev = np.linalg.norm(got["v"] - ref["v"], axis=1)
    assert np.all(ev[moving] <= 50 * TOL[prec] * vs[moving]), (ev / vs)[moving].max()
    m.close()
