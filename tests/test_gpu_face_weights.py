"""The FP64 face flux's HLL weights (double-float with an FP64 form behind it)
against the oracle, where their number range can go wrong: states scaled by
powers of two far outside binary32's range (the weights scale them back),
supersonic flow (one signal speed zero), the LLF option, and flat space at
radii where the squared speeds leave binary32's range (the FP64 form).
One CFL step; the bar is the FP64 path's, relative L1 1e-12 per field."""
import math

import numpy as np
import pytest

import oracle as O

from helpers import NG, gpu_grid, interior, rel_l1

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = (13, 6, 8)


def _smooth(n):
    k, j, i = np.meshgrid(*((np.arange(m) + 0.5) / m for m in (n[2], n[1], n[0])), indexing="ij")
    w = 2 * math.pi
    return (1 + 0.3 * np.sin(w * i) * np.cos(w * j), 0.8 + 0.2 * np.cos(w * (k + i)), 0.1 * np.sin(w * j),
            0.1 * np.cos(w * (i + k)), 0.1 * np.sin(w * (i - j)))


@pytest.mark.parametrize("scale,drift,riemann,r0", [
    (0, 0.3, O.FLUX_HLL, None),
    (-400, 0.3, O.FLUX_HLL, None),
    (400, 0.3, O.FLUX_HLL, None),
    (0, 4.0, O.FLUX_HLL, None),
    (0, -4.0, O.FLUX_HLL, None),
    (0, 0.3, O.FLUX_LLF, None),
    (-400, 0.3, O.FLUX_LLF, None),
    (0, 0.3, O.FLUX_HLL, 1e4),
    (0, 0.3, O.FLUX_HLL, 1e25),
])
def test_step_against_oracle(scale, drift, riemann, r0):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n1, n2, n3 = N
    rho, u, v1, v2, v3 = _smooth(N)
    s = 2.0 ** scale
    prim = np.zeros((8, n3 + 2 * NG, n2 + 2 * NG, n1 + 2 * NG))
    bf = np.zeros((3,) + prim.shape[1:])
    c = (slice(NG, NG + n3), slice(NG, NG + n2), slice(NG, NG + n1))
    if r0 is None:
        lo, h, metric, bc = (0.0, 0.0, 0.0), (1.0 / n1, 1.0 / n2, 1.0 / n3), O.METRIC_MINKOWSKI, (O.BC_PERIODIC,) * 6
        scales = (1.0, 1.0, 1.0)
        for d, b in enumerate((0.3, 0.2, -0.4)):  # a uniform field is divergence-free
            bf[d] = b * math.sqrt(s)
    else:
        lo, h, metric = (math.log(r0), 1.0, 0.0), (0.05, 1.0 / n2, 1.0 / n3), O.METRIC_SPHERICAL
        bc = (O.BC_OUTFLOW,) * 4 + (O.BC_PERIODIC,) * 2
        r = np.exp(lo[0] + (np.arange(n1) + 0.5) * h[0])[None, None, :]
        th = (lo[1] + (np.arange(n2) + 0.5) * h[1])[None, :, None]
        scales = (1 / r, 1 / r, 1 / (r * np.sin(th)))
    prim[0][c], prim[1][c] = s * rho, s * u
    for q, (v, sc) in enumerate(zip((v1 + drift, v2 - 0.2, v3 + 0.1), scales)):
        prim[2 + q][c] = v * sc
    d = O.make_desc(n1, n2, n3, *lo, *h, metric=metric, gam=5.0 / 3.0, cour=0.5, riemann=riemann, floors=0, bc=bc)
    g, og = gpu_grid(d), O.Grid(d)
    g.set_state(torch.from_numpy(prim).cuda(), torch.from_numpy(bf).cuda())
    og.set(prim, bf)
    st, dto = g.step(stats=True), og.step()
    pg, bg = g.get_state()
    po, bo = og.get()
    g.close()
    assert abs(st["dt_used"] - dto) <= 1e-12 * dto
    for q in (0, 1, 2, 3, 4):
        assert rel_l1(interior(pg[q], d), interior(po[q], d)) <= 1e-12, q
    if r0 is None:
        for q in range(3):
            assert rel_l1(interior(bg[q], d), interior(bo[q], d)) <= 1e-12, q
