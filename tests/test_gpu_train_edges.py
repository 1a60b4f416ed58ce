"""The training cluster at the edges of its row split: fewer rows than CTAs or than one 16-row tile,
whole and ragged chunks of 256 rows per CTA, more than one chunk, every input width class."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 4, 8])
@pytest.mark.parametrize("R", [1, 15, 16, 17, 255, 256, 257, 4096, 4097, 8192])
def test_first_step_takes_the_gradient_of_the_grad_kernel(D, R):
    import torch
    from paper_2311_12973_gb300 import smc2 as S
    rng = np.random.default_rng(100 * D + R)
    f32 = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    th, lp = f32(rng.standard_normal((R, D))), f32(-300 - 3 * rng.standard_normal(R) ** 2)
    p0 = f32(0.3 * rng.standard_normal(64 * D + 4289))
    p, m, v = p0.clone(), torch.zeros_like(p0), torch.zeros_like(p0)
    step = torch.zeros(1, dtype=torch.int32, device="cuda")
    x, y, _ = S.mlp_train_ring(p, m, v, step, th, lp, 0, 1e-3)
    assert torch.equal(p, p0) and int(step) == 0 and not m.any()
    x1, y1, z = S.mlp_train_ring(p, m, v, step, th, lp, 1, 1e-3)
    assert torch.equal(x, x1) and torch.equal(y, y1) and int(step) == 1
    loss, grad = S.mlp_loss_grad(p0, x, y)
    grad = grad.double().cpu().numpy()
    loss = float(loss)
    got = m.double().cpu().numpy() / float(np.float32(1) - np.float32(0.9))
    # The rows' terms are the same bits in both kernels; the sums over R rows differ in order only,
    # each off by at most R 2^-24 of its terms' magnitudes.  |h| <= 1 and sum |2 e / R| <= 2 sqrt(loss)
    # bound those: dw3 and db3 by s, dW2 and db2 by s |w3|, dW1 and db1 by s |w3| |W2|_1 |x|.
    w = p0.double().cpu().numpy()
    W2, w3 = w[64 * D + 64:64 * D + 4160].reshape(64, 64), w[64 * D + 4224:64 * D + 4288]
    s, a3 = 2.01 * np.sqrt(loss), np.abs(w3).max()
    back = s * np.abs(W2).sum(1).max() * a3 * 1.01
    terms = np.concatenate([np.full(64 * D, back * float(x.abs().max())), np.full(64, back), np.full(4160, s * a3),
                            np.full(65, s)])
    assert np.all(np.abs(got - grad) <= (2 * R + 8) * 2.0 ** -24 * terms)
    assert abs(z["loss"] - loss) <= (2 * R + 8) * 2.0 ** -24 * loss
