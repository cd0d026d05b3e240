"""The standalone inversion of batches at the edge between its two Newton forms (FP64 up to
one CTA of 128 states per SM, double-float with an FP64 last solve beyond): the same
states in batches below, at and above the edge give the oracle's outcomes and roots
within the bar that the conditioning of the inversion sets (helpers.inversion_bar)."""
import numpy as np
import pytest

import oracle as O
from helpers import inversion_bar
from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("over", [-1, 0, 1])
@pytest.mark.parametrize("network", [False, True])
def test_both_sides_of_the_edge(over, network):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    n = 128 * torch.cuda.get_device_properties(0).multi_processor_count + over
    pr, x1, x2 = W.random_states(n, seed=79, lorentz_range=(1.0, 10.0))
    g = pr.copy()
    g[:, 0] *= 1.05
    g[:, 1] *= 0.95
    g[:, 2:5] *= 1.02
    d = O.make_desc(1, 1, 1, 0, 0, 0, 1, 1, 1, metric=O.METRIC_KS, a=0.9375, gam=13.0 / 9.0)
    U = O.p2u_many(d, pr, x1, x2)
    want, so, _ = O.c2p_many(d, U, pr[:, 5:8], x1, x2, g)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    out = dev(g.T)
    st = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    net = hamr.Mlp(seed=7) if network else None  # as rescue: these starts need none
    hamr.con2prim(dev(U.T), dev(pr[:, 5:8].T), dev(x1), dev(x2), out, st, mlp=net, mlp_mode=hamr.MLP_RESCUE)
    out, st = out.cpu().numpy().T, st.cpu().numpy()
    if net is not None:
        net.close()
    assert (st == so).all()
    ok = so == 0
    assert ok.mean() > 0.999
    bar = inversion_bar(d, U[ok], pr[ok, 5:8], x1[ok], x2[ok], want[ok], pr[ok], p_other=out[ok])
    assert (np.abs(out[ok, :5] - want[ok, :5]) <= bar).all()
