"""The FP32 reconstruction's forms (one cell per thread; groups of two along x1 and
four along x2 and x3 on large launches) give the same bits: a block large enough
for the groups, whose sizes leave every remainder of a group, against the same
state cut into blocks that are too small for them is not comparable bit for bit,
so the large block is checked against the FP64 step at the mixed form's bar, and
its phi symmetry exactly: an axisymmetric state stays axisymmetric bit for bit
only if every cell of a group, at every place in it, takes the same arithmetic."""
import numpy as np
import pytest

from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [(97, 101, 66), (98, 102, 64), (99, 103, 64), (100, 100, 66)])
@pytest.mark.parametrize("recon", [0, 1, 2])
def test_groups_keep_axisymmetry_and_fp64_bar(n, recon):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    assert n[0] * n[1] * n[2] >= 152 * 4 * 8 * 32 * 4  # the groups' side of the rule
    geo = W.torus_geometry(*n)
    prim, bf = (torch.from_numpy(x).cuda() for x in W.torus_block(geo, pert=0.0))
    blk = hamr.block(*n, geo.x1min, geo.x2min, geo.x3min, geo.dx1, geo.dx2, geo.dx3, (3, 3, 2, 2, 1, 1))
    out = []
    for prec in (hamr.PREC_MIXED, hamr.PREC_FP64):
        g = hamr.Grid([blk], precision=prec, recon=recon)
        g.set_state(prim, bf)
        g.step()
        p, _ = g.get_state(prim=torch.empty_like(prim), bface=torch.empty_like(bf))
        out.append(p[:, 3:-3, 3:-3, 3:-3])
        g.close()
    mixed, fp64 = out
    assert torch.equal(mixed, mixed[:, :1].expand_as(mixed))
    # density after one step: FP32 unit round-off of the fluxes (6e-8) times dt/dx times the flux, below it
    assert (mixed[0] - fp64[0]).abs().sum() <= 6e-8 * fp64[0].abs().sum()
