"""Reading a state back on both sides of the size at which the copy changes (needs a GB300): small
states come in one copy through pinned memory, larger ones in one copy per array.  Checked: what is
stored exactly (groups, h and velocities in the working precision) comes back as it was loaded,
positions to the rounding of origin + cell edge + offset (the offset in the working precision), the
elements beyond the particles are zero, and single arrays may be left out."""
import ctypes as C

import numpy as np
import pytest

from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

PIN_BYTES = 256 * 1024


def staged(n):
    up = lambda b: (b + 255) // 256 * 256
    return 256 + 2 * up(24 * n) + up(8 * n) + 4 * n


MOST = max(n for n in range(1, 8192) if staged(n) <= PIN_BYTES)   # particles of the largest small state


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("n", [1, MOST, MOST + 1])
def test_round_trip(prec, n):
    w = WL.disk_holes(n_target=MOST + 400, seed=2, mc_samples=100_000)
    keep = np.sort(np.random.default_rng(5).permutation(len(w["x"]))[:n])
    w = WL.subset(w, keep)
    t = np.float32 if prec == 32 else np.float64
    h = (0.95 * WL.sizing_eval(w["sizing"], w["x"])).astype(t).astype(np.float64)
    v = np.zeros((n, 3))
    v[:, :2] = np.random.default_rng(6).normal(size=(n, 2)).astype(t)
    m = S.Mesh(w, precision=prec)
    m.set_state(v=v, h=h)
    got = S.sph_mesh_positions(m.h, n + 7)
    assert np.array_equal(got["group"][:n], w["group"])
    assert np.array_equal(got["h"][:n], h) and np.array_equal(got["v"][:n], v)
    c0 = float(S.sph_mesh_grid(m.h).c0)
    tol = (2.0 ** -24 * c0 if prec == 32 else 0.0) + 8 * np.finfo(float).eps * max(1.0, np.abs(w["x"]).max())
    assert np.abs(got["x"][:n] - w["x"]).max() <= tol
    assert all(not got[k][n:].any() for k in got)
    g = np.full(n, -1, np.int32)
    cnt = C.c_int64(0)
    assert S.lib().sph_mesh_positions(m.h, None, g.ctypes.data, None, None, n, C.addressof(cnt)) == 0
    assert cnt.value == n and np.array_equal(g, w["group"])
    m.close()
