"""The network's contractions at the edges of their tiles, against the FP64
reference with the same bf16 weights: widths that are no multiple of a tile or
of a 16-byte word, a single row, rows around a tile, and enough rows for the
large tiles; training steps apply the gradients that gradients() returns.
Tolerances as for the square network: fp32 sums of up to some hundred terms of
order one against FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup(torch, widths, B, seed):
    from paper_0705_0497_gb300 import api
    m = api.MLP(widths, seed=seed)
    rng = np.random.default_rng(seed + 1)
    X = rng.uniform(-1, 1, (B, widths[0])).astype(np.float32)
    T = (0.5 * np.sin(3.0 * X @ rng.standard_normal((widths[0], widths[-1])))).astype(np.float32)
    return m, X, T, torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()


@pytest.mark.parametrize("widths,B", [([4, 33, 257, 100], 1), ([3, 65, 31], 9), ([4, 64, 256, 864], 700),
                                      ([5, 257, 515, 863], 701), ([4, 300, 8], 64), ([8, 1], 3)])
def test_forward_and_gradients(torch_cuda, widths, B):
    import oracle.mlp_ref as R
    m, X, T, Xd, Td = _setup(torch_cuda, widths, B, seed=sum(widths) + B)
    p = m.params()
    Yr = R.forward(widths, p, X, bf16=True)[-1]
    assert np.max(np.abs(m.forward(Xd).cpu().numpy() - Yr)) <= 1e-5 * max(1.0, np.max(np.abs(Yr)))
    g, loss = m.gradients(Xd, Td)
    g = g.cpu().numpy()
    lr, gr = R.loss_and_grad(widths, p, X, T, bf16=True)
    assert abs(float(loss.item()) - lr) <= 1e-5 * lr
    lay, _ = R.layout(widths)
    for (ow, ob, a, b) in lay:
        for lo, hi in ((ow, ow + a * b), (ob, ob + b)):
            assert np.max(np.abs(g[lo:hi] - gr[lo:hi])) <= 1e-4 * np.max(np.abs(gr[lo:hi])) + 1e-12
    # one Adam step from rest: p - lr g / (|g| + eps) up to fp32 rounding
    m.train_step(Xd, Td, 1e-3)
    want = p - 1e-3 * g / (np.abs(g.astype(np.float64)) + 1e-8)
    assert np.max(np.abs(m.params() - want)) <= 2e-6 * max(1.0, np.max(np.abs(p)))
