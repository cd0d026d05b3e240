"""The FP64 face flux's HLL weights are FP64 numbers: between cells of independent
states (every face a jump of order one, all of it subsonic and in the energy
inversion's well-conditioned range) one step's conserved density rho Gamma is the
oracle's to rounding. The oracle's own distance from the same step in 80-bit
arithmetic is 1.7e-16 (rms, relative); two FP64 codes that round differently may
lie 2 to 3e-16 apart, the bar is 2^-51 = 4.4e-16. Weights of 46 bits, whose error
(5e-15) the jump multiplies, lie above it. The cells are narrow in one direction, so
that its fluxes carry the step (dt = 0.49 dx)."""
import math

import numpy as np
import pytest

import oracle as O

from helpers import NG, gpu_grid, interior

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("narrow", [0, 1, 2])
def test_jumps_to_rounding(narrow):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = [16, 16, 16]
    n[narrow] = 64
    h = [0.25, 0.25, 0.25]
    h[narrow] = 1.0 / 64
    n1, n2, n3 = n
    rng = np.random.default_rng(41 + narrow)
    prim = np.zeros((8, n3 + 2 * NG, n2 + 2 * NG, n1 + 2 * NG))
    bf = np.zeros((3,) + prim.shape[1:])
    c, s = (slice(NG, NG + n3), slice(NG, NG + n2), slice(NG, NG + n1)), (n3, n2, n1)
    prim[0][c] = np.exp(rng.uniform(math.log(0.1), 0.0, s))
    prim[1][c] = prim[0][c] * rng.uniform(0.3, 1.0, s)
    for q in (2, 3, 4):
        prim[q][c] = rng.uniform(-0.3, 0.3, s)
    for d, b in enumerate((0.3, 0.2, -0.4)):  # a uniform field is divergence-free
        bf[d] = b
    d = O.make_desc(n1, n2, n3, 0.0, 0.0, 0.0, *h, metric=O.METRIC_MINKOWSKI, gam=5.0 / 3.0, cour=0.5, floors=0,
                    bc=(O.BC_PERIODIC,) * 6)
    g, og = gpu_grid(d), O.Grid(d)
    g.set_state(torch.from_numpy(prim).cuda(), torch.from_numpy(bf).cuda())
    og.set(prim, bf)
    dt = og.step()
    g.step(dt)
    pg, po = interior(g.get_state()[0], d), interior(og.get()[0], d)
    g.close()

    def dens(p):
        return p[0] * np.sqrt(1.0 + p[2] ** 2 + p[3] ** 2 + p[4] ** 2)

    r = dens(pg) / dens(po) - 1.0
    assert math.sqrt((r * r).mean()) <= 2.0 ** -51
