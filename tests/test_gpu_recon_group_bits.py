"""The FP32 reconstruction's forms (one cell per thread on small launches; groups of two
cells along x1, four along x2 and x3 on large ones) give the same bits. A periodic box
in flat space with a random state goes through two steps of the mixed form; the same
state repeated several times in each direction fills a box that is large enough for
the groups: every repetition has to equal the small box bit for bit. The sizes leave
every remainder of a group in each direction, and the state varies in all three."""
import numpy as np
import pytest

from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

NG = 3
GROUPS_FROM = 152 * 4 * 8 * 32 * 4  # cells of a launch


def _state(n, seed):
    """Random periodic state of a box (no ghosts; faces 0..n-1), each B component constant along its own
    direction, so that its faces are divergence-free."""
    rng = np.random.default_rng(seed)
    s = (n[2], n[1], n[0])
    p = np.zeros((8,) + s)
    p[0] = np.exp(rng.uniform(-1.5, 0.0, s))
    p[1] = p[0] * rng.uniform(0.1, 1.0, s)
    p[2:5] = rng.uniform(-0.3, 0.3, (3,) + s)
    b = np.stack([np.broadcast_to(rng.uniform(-0.3, 0.3, [1 if d == ax else m for ax, m in enumerate(s)]), s)
                  for d in (2, 1, 0)])
    return p, b


def _padded(a):
    return np.pad(a, [(0, 0)] + [(NG, NG)] * 3, mode="wrap")


def _tiled(a, rep):
    return np.tile(a, (1, rep[2], rep[1], rep[0]))


def _advance(blocks, states, precision, dt, **kw):
    from paper_1912_10192_gb300 import hamr
    g = hamr.Grid([hamr.block_from_dict(b) for b in blocks], metric=hamr.METRIC_MINKOWSKI, gam=5.0 / 3.0, cour=0.5,
                  floors=0, precision=precision, **kw)
    if len(blocks) > 1:
        g.set_fine_dt(dt)
    out = []
    for i, (p, b) in enumerate(states):
        g.set_state(torch.from_numpy(_padded(p)).cuda(), torch.from_numpy(_padded(b)).cuda(), block=i)
    for _ in range(2):
        if len(blocks) > 1:
            g.batch_step(1)
        else:
            g.step(dt)
    for i in range(len(blocks)):
        p, b = g.get_state(block=i)
        out.append([a[:, NG:-NG, NG:-NG, NG:-NG] for a in (p, b)])
    g.close()
    return out


@pytest.mark.parametrize("n,rep", [((20, 18, 22), (5, 5, 4)), ((21, 19, 19), (5, 5, 5)), ((25, 21, 17), (3, 5, 5)),
                                   ((14, 16, 21), (7, 6, 6))])
@pytest.mark.parametrize("recon,flatten", [(0, 0), (0, 1), (1, 0), (2, 0)])
def test_single_block(n, rep, recon, flatten):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    p, b = _state(n, 5)
    big = [m * r for m, r in zip(n, rep)]
    assert np.prod(n) < GROUPS_FROM <= np.prod(big)
    h = 1.0 / 32
    mk = lambda m: [dict(n1=m[0], n2=m[1], n3=m[2], x1min=0.0, x2min=0.0, x3min=0.0, dx1=h, dx2=h, dx3=h,  # noqa: E731
                         bc=[1] * 6, lat=0)]
    kw = dict(recon=recon, flatten=flatten)
    small = _advance(mk(n), [(p, b)], hamr.PREC_MIXED, 0.2 * h, **kw)[0]
    large = _advance(mk(big), [(_tiled(p, rep), _tiled(b, rep))], hamr.PREC_MIXED, 0.2 * h, **kw)[0]
    assert not np.array_equal(small[0], p)
    for s, l in zip(small, large):
        assert np.array_equal(_tiled(s, rep), l)


@pytest.mark.parametrize("n,rep", [((15, 14, 17), (3, 3, 3)), ((13, 15, 16), (3, 3, 3)), ((12, 16, 15), (4, 3, 3)),
                                   ((17, 13, 14), (3, 4, 3))])
def test_tree(n, rep):
    """Eight blocks of one level, each with the same periodic content."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    p, b = _state(n, 6)
    assert 8 * np.prod(n) < GROUPS_FROM <= 8 * np.prod(n) * np.prod(rep)
    h = 1.0 / 32

    def blocks(m):
        out = W.flat_box_tree(base=(2, 2, 2), n=m, refine=(), lat_coarse=0)
        for x in out:
            for d in (1, 2, 3):  # cells of width h, whatever the block's size
                x["x%dmin" % d] *= h / x["dx%d" % d]
                x["dx%d" % d] = h
        return out

    small = _advance(blocks(n), [(p, b)] * 8, hamr.PREC_MIXED, 0.2 * h)
    large = _advance(blocks([m * r for m, r in zip(n, rep)]), [(_tiled(p, rep), _tiled(b, rep))] * 8,
                     hamr.PREC_MIXED, 0.2 * h)
    assert not np.array_equal(small[0][0], p)
    for s, l in zip(small, large):
        for x, y in zip(s, l):
            assert np.array_equal(_tiled(x, rep), y)
