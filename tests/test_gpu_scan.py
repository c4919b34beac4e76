"""The rebuild's counts and scan over many steps (needs a GB300): every step's scatter takes the
counts of the cells down to zero, on which the next step's histogram is built, and the scan looks
back over many tiles.  After steps, and after inspections that rebuild without stepping, the cell
starts are the exclusive sums of the keys' histogram and the permutation sorts the keys."""
import numpy as np
import pytest

from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def check(m):
    nc = S.sph_mesh_grid(m.h).n_cells
    key, cs, perm = S.sph_debug_rebuild(m.h, m.n, nc)
    assert np.array_equal(cs, np.concatenate([[0], np.cumsum(np.bincount(key, minlength=nc))]))
    assert np.array_equal(np.sort(perm), np.arange(m.n)) and (np.diff(key[perm]) >= 0).all()
    return nc


# one tile with a ragged end; a few tiles; more tiles than one look-back reads at once (128)
@pytest.mark.parametrize("shape,n,cps,cells", [("disk", 40, 1, 1), ("disk", 20_000, 2, 8 * 8192),
                                               ("cube", 60_000, 4, 128 * 8192)])
def test_cell_starts_over_steps(shape, n, cps, cells):
    make = WL.disk_holes if shape == "disk" else WL.cube_sphere
    w = make(n_target=n, seed=2, mc_samples=100_000)
    w["params"] = dict(w["params"], cells_per_support=cps)
    m = S.Mesh(w, precision=32)
    m.set_state()
    assert check(m) >= cells
    for k in (1, 3):
        m.step(k)
        m.sync()
        check(m)
        check(m)
    m.close()
