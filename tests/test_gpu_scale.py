"""Small domains (needs a GB300): the relaxation has no length of its own, so a 2D mesh of spacing
1e-10 in a domain of 2e-9 gives the accelerations of the oracle and stays finite, as far as h^4, the
smallest power the single-precision sums hold, is a number at all."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def scaled(w, k):
    """The problem with every length times k."""
    dom, siz = dict(w["domain"]), w["sizing"]
    dom["lo"], dom["hi"] = [k * v for v in dom["lo"]], [k * v for v in dom["hi"]]
    dom["features"] = [{q: [k * t for t in v] if q in ("a", "b", "p") else v for q, v in f.items()} for f in dom["features"]]
    siz = dict(siz, **{q: k * siz[q] for q in ("a", "lo", "hi")})
    return dict(w, domain=dom, sizing=siz, x=k * w["x"], h_lo=k * w["h_lo"], h_hi=k * w["h_hi"])


@pytest.mark.parametrize("k", [1.0, 2e-8, 2e-9])
def test_small_2d_domains(k):
    w = scaled(WL.square2d(h=0.05), k)
    h = O.Oracle(w).h.astype(np.float32).astype(np.float64)
    o = O.Oracle(w, h=h)
    ref = o.interact()
    m = S.Mesh(w, precision=32)
    m.set_state(h=h)
    got = S.sph_debug_interact(m.h, m.n, m.n_groups)
    # the pressure pass's bound, and the spacing of the single-precision numbers at h^4
    tol = 1e-5 + np.spacing(np.float32(h.min() ** 4)) / h.min() ** 4
    err = np.linalg.norm(got["a_p"] - ref["a_p"], axis=1)
    assert np.all(err <= tol * ref["S"]), (err / np.maximum(ref["S"], 1e-300)).max()
    m.step(20)
    m.sync()
    p = m.positions()
    assert np.isfinite(p["x"]).all() and np.isfinite(p["v"]).all()
    assert np.abs(p["x"] - w["x"]).max() > 0
    m.close()
