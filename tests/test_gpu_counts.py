"""Target counts where rounding decides (needs a GB300): with a constant spacing the integral of h^-d
over an edge, a face or a box is often an odd multiple of 1/2, and the rounding of its terms and the
order of their sum decide the count.  Both are part of the result: the integrals equal, bit for bit,
the same sum done here (equal terms measure / nq^d / h^d, divided once; 608 blocks of 256 threads
stride over the points, each thread adds its terms one by one, a warp's lanes are added in halves,
the warps and then the blocks in order)."""
import numpy as np
import pytest

from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S

pytestmark = pytest.mark.gpu

BLOCKS, THREADS = 608, 256


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def total(term, npts):
    share = np.maximum(0, -((np.arange(BLOCKS * THREADS) - npts) // (BLOCKS * THREADS)))
    sums = np.concatenate([[0.0], np.add.accumulate(np.full(share.max(), term))])
    v = sums[share].reshape(BLOCKS, THREADS // 32, 32)
    while v.shape[2] > 1:
        half = v.shape[2] // 2
        v = v[:, :, :half] + v[:, :, half:]
    warps = v[:, :, 0]
    block = np.zeros(BLOCKS)
    for w in range(warps.shape[1]):
        block = block + warps[:, w]
    return np.add.accumulate(block)[-1]


def box(D, L):
    feats = [dict(kind="volume", dim=D)]
    for a in range(D):
        e = [0.0, 0.0, 0.0]
        e[a] = L[a]
        feats.append(dict(kind="segment", dim=1, a=[0.0, 0.0, 0.0], b=e, nb=[1.0, 0.0, 0.0]))
    if D == 3:
        for a in range(3):
            u, w = [0.0] * 3, [0.0] * 3
            u[a], w[(a + 1) % 3] = 1.0, 1.0
            feats.append(dict(kind="rect", dim=2, o=[0.0, 0.0, 0.0], u=u, w=w, lu=L[a], lw=L[(a + 1) % 3],
                              nb=[0.0, 0.0, 1.0]))
    return dict(D=D, base="box", lo=[0.0, 0.0, 0.0], hi=list(L[:D]) + [0.0] * (3 - D), ball_c=[0, 0, 0],
                ball_r=0.0, holes=[], features=feats)


def expected(D, L, h):
    nv = 2048 if D == 2 else 256
    cell = 1.0
    for a in range(D):
        cell *= L[a] / nv
    out = [total(cell / (h * h if D == 2 else h * h * h), nv ** D)]
    out += [total(np.sqrt(L[a] * L[a]) / 65536 / h, 65536) for a in range(D)]
    if D == 3:
        out += [total((L[a] / 1024) * (L[(a + 1) % 3] / 1024) / (h * h), 1024 ** 2) for a in range(3)]
    return np.array(out)


# one sizing per kind, all of them constant over the domain
@pytest.mark.parametrize("kind", ["const", "radial", "hole_dist"])
@pytest.mark.parametrize("D", [2, 3])
def test_counts_at_odd_halves(D, kind):
    rng = np.random.default_rng(17 + D)
    ties = 0
    for h in (0.1, 0.2, 0.05, 0.04, 0.03, 0.07, 0.013):
        for _ in range(4):
            L = [float((int(rng.integers(3, 40)) + 0.5) * h) for _ in range(D)]
            refs = [([0.1, 0.2, 0.0], 0.05), ([0.9, 0.7, 0.0], 0.1)] if kind == "hole_dist" else []
            siz = dict(kind=kind, a=h, b=0.0, lo=h, hi=2 * h if kind == "hole_dist" else h, q=[0, 0, 0], refs=refs)
            M, N = S.sph_feature_counts(S.domain_desc(box(D, L)), S.sizing_desc(siz))
            ref = expected(D, L, h)
            assert np.array_equal(M, ref), (h, L, M - ref)
            assert np.array_equal(N, np.floor(ref + 0.5).astype(np.int64))
            ties += int((np.abs(ref - np.floor(ref) - 0.5) < 1e-10).sum())
    assert ties > 50   # the case is met
