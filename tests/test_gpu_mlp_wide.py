"""The control's network with a wide input layer, whose tiles shrink to fit the shared memory: gradient
and loss against the FP64 oracle, at the widths around each limit (255 / 256 inputs for 64 samples a
tile) and the widest that fits at all, one training step beside them.  Tolerance as for the narrow ones: rounding of a mean of M products in
FP32, with the sum over the inputs in the first layer: 2^-24 (64 + nin + tiles / 16 + 16) times 4."""
import numpy as np
import pytest

from oracle import learned as Lr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,M", [(255, 19457), (256, 19457), (288, 19457), (288, 4865)])
def test_wide_input_layer(nin, M):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_19171_gb300 as P
    rng = np.random.default_rng(nin)
    p = np.float64(np.float32(Lr.init_params(nin, seed=3)))
    x = np.float64(np.float32(rng.uniform(-1, 1, (M, nin))))
    y = np.float64(np.float32(np.stack([rng.uniform(0.01, 0.4, M), rng.uniform(2, 6, M)], 1)))
    loss, g = Lr.loss_and_grad(p, x, y, 7)
    t = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    l2, g2 = P.mlp_grad(t(p), t(x), t(y), 7)
    tol = 4 * 2.0 ** -24 * (64 + nin + M / 64 / 16 + 16)
    assert abs(l2 - loss) <= tol
    assert np.abs(g2.cpu().numpy() - g).max() <= tol
    out = P.mlp_forward(t(p), t(x), 7, bf16=False).cpu().numpy()
    gam, kc = Lr.outputs_to_filter(Lr.forward(p, x)[0], 7)
    assert np.abs(out[:, 0] - gam).max() <= 1e-5 and np.abs(out[:, 1] - kc).max() <= 1e-4
    q = t(p)
    m, v = torch.zeros_like(q), torch.zeros_like(q)
    hist, steps = P.mlp_train(q, m, v, t(x), t(y), 7, batch=M, epochs=1, lr=1e-3)
    assert steps == 1 and abs(hist[0] - loss) <= tol
