"""The training loss of a large batch against 64 bits. It is a running FP32 sum whose terms
arrive in any order, so its rounding grows with the number of terms: 1.6e-6 (rms,
relative; simulated) for sums over 16 samples of a batch of 2^18, 1.3e-6 over 32, 8e-7
over a CTA's 64. The bar lies between the last two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_loss_of_a_large_batch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_10192_gb300 import hamr
    n, reps = 1 << 18, 96
    gen = torch.Generator(device="cuda").manual_seed(4)
    m = hamr.Mlp(seed=7)
    err = []
    for _ in range(reps):
        feat = torch.randn((10, n), generator=gen, device="cuda")
        targ = torch.randn((2, n), generator=gen, device="cuda")
        m.fit_norm(feat, targ)
        loss, _ = m.loss_grad(feat, targ)
        p, nrm = (torch.from_numpy(a).cuda().double() for a in m.params())
        h, o = (feat.double().T - nrm[:10]) / nrm[10:20], 0
        for rows, cols in ((64, 10), (64, 64), (64, 64), (2, 64)):
            h = h @ p[o:o + rows * cols].view(rows, cols).T + p[o + rows * cols:o + rows * cols + rows]
            o += rows * cols + rows
            if rows == 64:
                h = torch.tanh(h)
        want = float(((h - (targ.double().T - nrm[20:22]) / nrm[22:24]) ** 2).sum()) / (2 * n)
        err.append(loss / want - 1.0)
    m.close()
    assert np.sqrt(np.mean(np.square(err))) <= 1.05e-6
