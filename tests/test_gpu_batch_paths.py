"""An instance alone and in a batch where the two take different kernels (needs a GB300): the kernels of
the update and the width of the search follow the slots of the whole batch, and the width in 2D the
levels of its grids; results do not.  Positions, velocities and spacings are compared bit for bit after
a few steps (velocities carried from the second on)."""
import numpy as np
import pytest

from paper_2003_01061_gb300 import build as B
from paper_2003_01061_gb300 import sphmesh as S
from paper_2003_01061_gb300 import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    B.build()


def make(shape, n, seed):
    if shape == "square":   # one grid level
        return WL.square2d(h=1.0 / round(n ** 0.5 - 1), seed=seed)
    return (WL.disk_holes if shape == "disk" else WL.cube_sphere)(n_target=n, seed=seed, mc_samples=50_000)


# (instances, steps, precision).  2D: three update kernels beyond 65,536 slots, a search for 8 beyond
# 65,536 and for 16 beyond 524,288, on one level beyond 32,768 and 262,144; 3D: three kernels beyond
# 8,192 slots, a search for 4, 8 and 16 beyond 32,768, 65,536 and 524,288
@pytest.mark.parametrize("parts,steps,prec", [
    ([("disk", 36_000), ("disk", 34_000)], 8, 32),
    ([("disk", 270_000), ("disk", 270_000)], 4, 32),
    ([("square", 20_000), ("square", 20_000)], 8, 32),
    ([("square", 30_000), ("disk", 4_000)], 8, 32),
    ([("square", 140_000), ("square", 140_000), ("square", 2_600)], 5, 32),
    ([("disk", 20_000), ("disk", 50_000)], 5, 64),
    ([("cube", 6_000), ("cube", 5_000)], 10, 32),
    ([("cube", 20_000), ("cube", 18_000)], 6, 32),
    ([("cube", 40_000), ("cube", 30_000)], 6, 32),
    ([("cube", 270_000), ("cube", 260_000)], 3, 32)])
def test_alone_and_batched_bit_for_bit(parts, steps, prec):
    ws = [make(s, n, 3 + i) for i, (s, n) in enumerate(parts)]
    b = S.Batch(ws, precision=prec)
    for i in range(len(ws)):
        b.set_state(i)
    b.step(steps)
    b.sync()
    for i, w in enumerate(ws):
        m = S.Mesh(w, precision=prec)
        m.set_state()
        m.step(steps)
        m.sync()
        p, q = m.positions(), b.positions(i)
        m.close()
        for k in ("x", "v", "h", "group"):
            assert np.array_equal(p[k], q[k]), (parts[i], k, (p[k] != q[k]).sum())
    b.close()
