"""A state loaded from and read into device memory (one kernel each) against the
host-memory calls (runtime copies): the same bits over the whole padded block,
before and after a step, at sizes that end a CTA and a warp raggedly, for a
single block and for the blocks of a tree."""
import numpy as np
import pytest

from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _grids(kind):
    from paper_1912_10192_gb300 import hamr
    if kind == "tree":
        blocks = W.flat_box_tree(base=(2, 1, 1), n=(5, 4, 7), refine=((0, 0, 0),), lat_coarse=1, lat_fine=0)
        mk = lambda: hamr.Grid([hamr.block_from_dict(b) for b in blocks], metric=hamr.METRIC_MINKOWSKI,  # noqa: E731
                               gam=5.0 / 3.0, cour=0.5, floors=0)
        return mk, W.flat_box_state(blocks), lambda g: g.batch_step(2)
    geo = W.torus_geometry(*kind)
    blk = hamr.block(*kind, geo.x1min, geo.x2min, geo.x3min, geo.dx1, geo.dx2, geo.dx3, (3, 3, 2, 2, 1, 1))
    return (lambda: hamr.Grid([blk])), [W.torus_block(geo, seed=3)], lambda g: g.step()


@pytest.mark.parametrize("kind", [(4, 4, 4), (17, 9, 6), (58, 21, 10), "tree"])
def test_device_and_host_calls_agree(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mk, states, step = _grids(kind)
    host, dev = mk(), mk()
    for b, (p, f) in enumerate(states):
        host.set_state(p, f, block=b)
        dev.set_state(torch.from_numpy(p).cuda(), torch.from_numpy(f).cuda(), block=b)
    for _ in range(2):
        for b, (p, f) in enumerate(states):
            ph, fh = host.get_state(block=b)
            pd, fd = torch.full(p.shape, -7.0, dtype=torch.float64, device="cuda"), torch.empty_like(torch.from_numpy(f)).cuda()
            dev.get_state(block=b, prim=pd, bface=fd)
            assert np.array_equal(ph, pd.cpu().numpy()) and np.array_equal(fh, fd.cpu().numpy())
        step(host)
        step(dev)
    host.close()
    dev.close()
