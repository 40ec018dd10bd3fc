"""Gradient, loss and inference of the control's network at sample counts around every change of the
tile size (8, 16, 32, 64 samples a tile) and with part-filled last tiles, against the FP64 oracle.
A gradient entry is a mean of M products in FP32: its rounding stays below 2^-24 (64 + tiles / 16 + 16)
times the mean of the products' magnitudes, which the test bounds by 4 (targets and weights of
order one)."""
import numpy as np
import pytest

from oracle import learned as Lr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2509_19171_gb300 import build
    build.build()
    import paper_2509_19171_gb300 as pkg
    return pkg


@pytest.mark.parametrize("N,M", [(7, 1), (7, 7), (5, 1216), (7, 1217), (6, 4865), (9, 19457)])
def test_gradient_and_forward(P, N, M):
    import torch
    nin = 2 * (N + 1)
    rng = np.random.default_rng(M)
    p = np.float64(np.float32(Lr.init_params(nin, seed=3)))
    x = np.float64(np.float32(rng.uniform(-1, 1, (M, nin))))
    y = np.float64(np.float32(np.stack([rng.uniform(0.01, 0.4, M), rng.uniform(2, N - 1, M)], 1)))
    loss, g = Lr.loss_and_grad(p, x, y, N)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    l2, g2 = P.mlp_grad(t(p), t(x), t(y), N)
    tol = 4 * 2.0 ** -24 * (64 + M / 64 / 16 + 16)
    assert abs(l2 - loss) <= tol
    assert np.abs(g2.cpu().numpy() - g).max() <= tol
    o, _ = Lr.forward(p, x)
    gam, kc = Lr.outputs_to_filter(o, N)
    out = P.mlp_forward(t(p), t(x), N, bf16=False).cpu().numpy()
    assert np.abs(out[:, 0] - gam).max() <= 1e-5 and np.abs(out[:, 1] - kc).max() <= 1e-4
