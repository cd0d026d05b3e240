"""The geometry kernels (twelve threads per point on small planes, one on large ones) give
the same tables: a small block and a large one that share their lower corner in x1 and x2
and so their first points take one step of the same state; the cells that the other
boundaries have not reached have to agree at the FP64 path's bar (relative L1 1e-12)."""
import numpy as np
import pytest

from helpers import rel_l1
from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NG = 3


@pytest.mark.parametrize("bc2", [(2, 0), (0, 0)])  # a polar axis at the shared corner, or none
@pytest.mark.parametrize("small", [(40, 30), (17, 13)])
def test_small_and_large_planes(bc2, small):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    n1, n2, n3 = 130, 64, 8
    m1, m2 = small
    assert (m1 + 6) * (m2 + 6) < 6144 <= (n1 + 6) * (n2 + 6)
    geo = W.torus_geometry(n1, n2, n3)
    prim, bf = W.torus_block(geo, seed=9)
    prim[1, :] *= 1.0 + 0.1 * np.random.default_rng(2).uniform(-1, 1, prim[1].shape)
    x2min = geo.x2min if bc2[0] == 2 else 0.3
    out = []
    for a1, a2 in ((n1, n2), small):
        blk = hamr.block(a1, a2, n3, geo.x1min, x2min, geo.x3min, geo.dx1, 0.9 * geo.dx2, geo.dx3,
                         (3, 0) + bc2 + (1, 1))
        g = hamr.Grid([blk])
        cut = (slice(None), slice(None), slice(0, a2 + 2 * NG), slice(0, a1 + 2 * NG))
        g.set_state(np.ascontiguousarray(prim[cut]), np.ascontiguousarray(bf[cut]))
        g.step(1e-3)
        out.append(g.get_state()[0][:, NG:-NG, NG:NG + m2 - 2 * NG, NG:NG + m1 - 2 * NG])
        g.close()
    big, sml = out
    assert not np.array_equal(big[0], prim[0, NG:-NG, NG:NG + m2 - 2 * NG, NG:NG + m1 - 2 * NG])
    for q in range(8):
        assert rel_l1(sml[q], big[q]) <= 1e-12, q
