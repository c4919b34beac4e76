"""Domains of millions of cells along x (needs a GB300).  The search keeps positions in single precision,
modulo 16,384 cells along x: around the places where that starts again, at the domain's start and at
its end, the neighbour sets equal brute force on the stored representation, and the search looks at as
many candidates as at the start."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

WRAP = 1 << 14


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def ribbon(D, cells, levels, spots):
    """A thin domain with a patch of particles around each of the cell coordinates `spots`: the problem,
    the smoothing lengths and the particles' patches."""
    h, ratio = 0.01, 2 ** (levels - 1)
    og = O.grid_spec(D, [0, 0, 0], [1, 1, 1 if D == 3 else 0], h, ratio * h, kappa=2.6, cells_per_support=2)
    c0, lead, side = float(og.c0), -float(og.origin[0]), 6 * h * ratio
    dom = dict(D=D, base="box", lo=[0.0, 0.0, 0.0], hi=[cells * c0, side, side if D == 3 else 0.0], ball_c=[0, 0, 0],
               ball_r=0.0, holes=[], features=[dict(kind="volume", dim=D)])
    siz = dict(kind="radial", a=h, b=0.2 if ratio > 1 else 0.0, lo=h, hi=ratio * h, q=[0, 0, 0], refs=[])
    rng, n = np.random.default_rng(7), 150 if D == 2 else 400
    x = np.zeros((len(spots), n, 3))
    x[:, :, :D] = rng.random((len(spots), n, D)) * side
    x[:, :, 0] += (np.array(spots) * c0 - lead - 0.5 * side)[:, None]
    hs = (h * ratio ** rng.random(x.shape[:2])).astype(np.float32).astype(np.float64)
    keep = (x[:, :, 0] > 0) & (x[:, :, 0] < cells * c0)
    patch = np.nonzero(keep)[0]
    return dict(name="ribbon", domain=dom, sizing=siz, params=dict(WL.PAPER_PARAMS), x=x[keep],
                group=np.zeros(len(patch), np.int32), h_lo=h, h_hi=ratio * h), hs[keep], patch


@pytest.mark.parametrize("D,levels,log_cells", [(2, 1, 22), (2, 4, 20), (3, 2, 18)])
@pytest.mark.parametrize("prec", [32, 64])
def test_neighbor_sets_along_a_long_domain(D, levels, log_cells, prec):
    cells = (1 << log_cells) - 200
    spots = [30, WRAP // 4, WRAP, 3 * WRAP // 4 + 5 * WRAP, 7 * WRAP + 3, cells // WRAP * WRAP, cells]
    w, h, patch = ribbon(D, cells, levels, spots)
    m = S.Mesh(w, precision=prec)
    m.set_state(h=h)
    g = S.sph_mesh_grid(m.h)
    assert g.levels == levels and g.dims[0][0] > cells
    og = O.grid_spec(D, w["domain"]["lo"], w["domain"]["hi"], w["h_lo"], w["h_hi"], kappa=2.6,
                     cells_per_support=g.cells_per_support)
    for mode in (0, 1):
        counts, lists = S.sph_debug_neighbors(m.h, m.n, mode)
        off = np.concatenate([[0], np.cumsum(counts)])
        for i in range(m.n):
            ref = O.neighbors_repr(og, w["x"], h, i, prec=prec, kappa=2.6, self_radius=mode == 1)
            assert np.array_equal(lists[off[i]:off[i + 1]], ref), (i, w["x"][i])
    far = S.sph_debug_pair_counts(m.h)
    m.close()
    # every patch by itself, moved to the first cells of a short domain by whole top-level cells
    top, near = 2 ** (levels - 1) * float(g.c0), [0, 0]
    for s in range(len(spots)):
        x = w["x"][patch == s].copy()
        x[:, 0] -= (np.floor(x[:, 0].min() / top) - 8) * top
        v = dict(w, x=x, group=w["group"][patch == s], domain=dict(w["domain"], hi=[200 * top] + w["domain"]["hi"][1:]))
        m = S.Mesh(v, precision=prec)
        m.set_state(h=h[patch == s])
        near = [a + b for a, b in zip(near, S.sph_debug_pair_counts(m.h))]
        m.close()
    assert abs(far[1] - near[1]) <= 4   # pairs at the support's edge, by the rounding of the move
    assert far[0] <= 1.1 * near[0], (far, near)

