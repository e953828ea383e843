"""The surrogate's kernels at the edges of their tiles (128 positions per stage
and 32 per step in layer 1, 128 tours per head tile and per slab of the gradient
kernel; more tours than two lines of 152 CTAs take in one turn), against the
FP64 reference with the tolerances of the other surrogate tests."""
import numpy as np
import pytest

from oracle import mlp_reference as M
from synth import make_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,n", [(1, 1), (17, 31), (127, 33), (129, 128), (305, 129), (1300, 40), (3, 1100)])
def test_forward_and_gradients(T, n):
    import paper_2511_18022_gb300 as cv
    from paper_2511_18022_gb300 import build
    build.build()
    rng = np.random.default_rng([T, n])
    inst = make_instance(n, 5, 20, seed=T + n, Q=64)
    cust = np.column_stack([inst.coords[1:, 0], inst.coords[1:, 1], rng.integers(5, 21, n),
                            rng.integers(1, 6, n)]).astype(np.float32)
    tours = np.stack([rng.permutation(n) + 1 for _ in range(T)]).astype(np.int32)
    target = rng.normal(size=T).astype(np.float32)
    sp = cv.Splitter(0)
    sur = cv.Surrogate(sp.ctx, cust, inst.dist, Q=64.0, seed=3)
    p = sur.params()
    phi, t = M.features(tours, cust, inst.dist, Q=64.0)   # Q = 2^6 keeps the features exact in fp32
    wloss, wg, want = M.loss_and_grad(p, phi, t, target, bf16=True)
    dev = torch.from_numpy(tours).cuda()
    out = torch.empty(T, dtype=torch.float32, device="cuda")
    sur.predict(dev, out)
    assert np.allclose(out.cpu().numpy(), want, rtol=1e-4, atol=1e-4)
    g, loss = sur.gradients(dev, torch.from_numpy(target).cuda())
    assert abs(loss - wloss) <= 1e-4 * max(1.0, wloss)
    for lo, hi in ((M.OFF_W1, M.OFF_B1), (M.OFF_B1, M.OFF_W2), (M.OFF_W2, M.OFF_B2), (M.OFF_B2, M.OFF_W3),
                   (M.OFF_W3, M.OFF_B3), (M.OFF_B3, M.NPARAMS)):
        scale = np.abs(wg[lo:hi]).max() + 1e-12
        assert np.abs(g[lo:hi] - wg[lo:hi]).max() <= 1e-3 * scale, (lo, hi)
    sur.close()
    sp.close()
