"""The learned guess's products at the edges of their 64 x 64 x 32 tiles and minibatch splits (1, 63 to 65, 127 to 129
rows, odd sizes, more rows than one split takes), with 16-byte aligned and unaligned inputs, against the FP64 network of
the oracle on the same bfloat16 weights.

Every sum has at most 2,049 FP32 terms in tiles of 32: rounding of order sqrt(2049) * 6e-8 = 3e-6 of the terms'
magnitude, of which the largest gradient element is at least a twentieth part here: 1e-4 of it bounds the error."""
import numpy as np
import pytest

from paper_1708_00033_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,shift", [(1, 0), (31, 1), (63, 0), (64, 0), (65, 3), (127, 0), (129, 0), (255, 1), (1000, 0), (2049, 0)])
def test_training_step_sizes(n, shift):
    import torch

    from oracle import mlp
    from paper_1708_00033_gb300 import hf
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 16)).astype(np.float32)
    T = rng.normal(size=(n, 325)).astype(np.float32)
    M = (rng.random((n, 325)) < 0.4).astype(np.float32)
    w = inputs.guess_init_weights(n)
    wb, o = w.astype(np.float64), 0
    for s in mlp.SHAPES:  # matrices enter the products as bfloat16
        k = int(np.prod(s))
        if len(s) == 2:
            wb[o:o + k] = mlp.to_bf16(w[o:o + k])
        o += k
    loss_ref, g_ref = mlp.loss_and_grad(wb, X, T, M)
    Y_ref, _ = mlp.forward(wb, X)
    flat = torch.zeros(16 * n + shift, dtype=torch.float32, device="cuda:0")
    Xd = flat[shift:].view(n, 16)  # a view that starts `shift` floats into an allocation
    Xd.copy_(torch.from_numpy(X))
    model = hf.Model(hf.Context(0), w)
    Y = model.forward(Xd).cpu().numpy()
    assert np.abs(Y - Y_ref).max() <= 1e-4 * np.abs(Y_ref).max()
    loss = model.train_step(Xd, torch.from_numpy(T).cuda(), torch.from_numpy(M).cuda(), lr=0.0)
    g = model.weights(gradients=True)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    assert np.abs(g - g_ref).max() <= 1e-4 * np.abs(g_ref).max()
