"""Device pointers that no kernel can take go through the runtime's copies: a
state at an address that is no multiple of eight bytes loads and reads out with the
same bits, and an allocation one value too short is refused with an error, the
device still usable after it. (The short allocation ends inside a mapped page, so
that nothing here depends on the refusal to stay in bounds.)"""
import ctypes as C

import numpy as np
import pytest

from paper_1912_10192_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = (11, 6, 8)


def _grid_and_state():
    from paper_1912_10192_gb300 import hamr
    geo = W.torus_geometry(*N)
    g = hamr.Grid([hamr.block(*N, geo.x1min, geo.x2min, geo.x3min, geo.dx1, geo.dx2, geo.dx3, (3, 3, 2, 2, 1, 1))])
    return g, W.torus_block(geo, seed=3)


def _at(a, shift):
    """A copy of the array's bytes on the device, `shift` bytes into a buffer."""
    buf = torch.zeros(a.nbytes + 16, dtype=torch.uint8, device="cuda")
    buf[shift:shift + a.nbytes] = torch.from_numpy(a.reshape(-1).view(np.uint8)).cuda()
    return buf


@pytest.mark.parametrize("shift", [0, 1, 4, 8])
def test_any_alignment(shift):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    g, (prim, bf) = _grid_and_state()
    g.set_state(prim, bf)
    want = g.get_state()
    p, b = _at(prim, shift), _at(bf, shift)
    hamr.check(hamr.lib().hamr_grid_set_state(g.h, 0, p.data_ptr() + shift, b.data_ptr() + shift, 1, None))
    po, bo = _at(np.zeros_like(prim), shift), _at(np.zeros_like(bf), shift)
    hamr.check(hamr.lib().hamr_grid_get_state(g.h, 0, po.data_ptr() + shift, bo.data_ptr() + shift, 1, None))
    for buf, a in ((po, want[0]), (bo, want[1])):
        raw = buf.cpu().numpy()
        assert np.array_equal(raw[shift:shift + a.nbytes], a.reshape(-1).view(np.uint8))
        assert not raw[:shift].any() and not raw[shift + a.nbytes:].any()
    g.close()


def test_short_allocation_is_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    g, (prim, bf) = _grid_and_state()
    g.set_state(torch.from_numpy(prim).cuda(), torch.from_numpy(bf).cuda())
    want = g.get_state()
    cu = C.CDLL("libcuda.so.1")
    ptr = C.c_uint64()
    assert prim.nbytes < 1 << 20 and cu.cuMemAlloc_v2(C.byref(ptr), C.c_size_t(prim.nbytes - 8)) == 0
    b = torch.from_numpy(bf).cuda()
    for call in (hamr.lib().hamr_grid_get_state, hamr.lib().hamr_grid_set_state):
        assert call(g.h, 0, ptr.value, b.data_ptr(), 1, None) != 0
    torch.cuda.synchronize()
    g.set_state(torch.from_numpy(prim).cuda(), torch.from_numpy(bf).cuda())
    got = g.get_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    g.close()
    assert cu.cuMemFree_v2(ptr) == 0


def test_under_capture():
    """A load and a read-out captured into a graph, with the pointers asked about during the capture."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g, (prim, bf) = _grid_and_state()
    p, b = torch.from_numpy(prim).cuda(), torch.from_numpy(bf).cuda()
    po, bo = torch.zeros_like(p), torch.zeros_like(b)
    g.set_state(p, b)
    want = g.get_state()
    s, gr = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(gr, stream=s):
        g.set_state(p, b, stream=s)
        g.get_state(prim=po, bface=bo, stream=s)
    gr.replay()
    torch.cuda.synchronize()
    assert np.array_equal(po.cpu().numpy(), want[0]) and np.array_equal(bo.cpu().numpy(), want[1])
    g.close()
