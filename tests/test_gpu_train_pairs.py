"""The fused training pass at the edges of its 128-row tiles and of the weight gradients' 64-row slices, against the
FP64 loss and gradient with the same BF16 roundings (the bounds of the other network tests)."""
import numpy as np
import pytest

import oracle
from oracle import mlp_oracle as mo
from paper_2510_16172_gb300 import fpt
from test_gpu_mlp import SCALE, numpy_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2510_16172_gb300 import build

    build.build()
    oracle.build()
    return fpt.Context(0)


@pytest.mark.parametrize("n,shift", [(1, 0), (63, 0), (127, 1), (129, 0), (200, 0), (9729, 0), (19_531, 1)])
def test_gradient_at_tile_edges(ctx, n, shift):
    """shift: the samples start one element into their buffers, so that nothing is 16-byte aligned."""
    import torch

    rng = np.random.default_rng(n)
    Xo = mo.bf16(rng.uniform(-1.0, 1.0, (n, 64)))
    G = rng.normal(0.0, 1.0, (n, 4, 3))
    T = rng.uniform(-0.5, 1.5, (n, 8))
    params = numpy_params(8)
    net = fpt.Mlp(ctx, 0, SCALE)
    net.set_params(params)

    def put(a, dtype):
        buf = torch.zeros(a.size + shift, dtype=dtype, device="cuda")
        buf[shift:] = torch.as_tensor(a, dtype=torch.float32).to(dtype).cuda().reshape(-1)
        return buf[shift:].view(a.shape)

    loss, g = net.loss_grad(put(Xo, torch.bfloat16), put(T, torch.float32), put(G, torch.float32))
    lo, go = mo.loss_grad(params.astype(np.float64), Xo, T, G)
    assert abs(loss - lo) <= 2e-3 * abs(lo)
    g = g.cpu().numpy()
    assert np.abs(g - go).max() <= 3e-3 * np.abs(go).max(), (np.abs(g - go).max(), np.abs(go).max())
    net.close()


def test_chained_steps_equal_single_steps(ctx):
    """The steps of one fpt_mlp_train call start from the gradient the step before cleared and overlap it; single steps
    (fpt_mlp_train_step) clear it themselves and do not.  Batches of the whole set, so that every step sees the same samples: 6
    chained epochs against 6 single steps, weights within a few learning rates where a gradient changes sign with the
    order of the sums (Adam's first steps move a weight by +-lr), equal to 1e-3 lr almost everywhere."""
    import torch

    rng = np.random.default_rng(3)
    n, lr = 384, 1e-3
    X = torch.as_tensor(rng.uniform(-1.0, 1.0, (n, 64)), dtype=torch.float32).to(torch.bfloat16).cuda()
    T = torch.as_tensor(rng.uniform(-0.5, 1.5, (n, 8)), dtype=torch.float32, device="cuda")
    G = torch.as_tensor(rng.normal(0.0, 1.0, (n, 12)) ** 2, dtype=torch.float32, device="cuda")
    a, b = fpt.Mlp(ctx, 7, SCALE), fpt.Mlp(ctx, 7, SCALE)
    hist = a.train(X, T, G, epochs=6, batch=n, lr=lr, lr_decay=1.0, seed=3)
    losses = [b.train_step(X, T, G, lr) for _ in range(6)]
    np.testing.assert_allclose(hist, losses, rtol=1e-4)
    diff = np.abs(a.get_params() - b.get_params())
    assert diff.max() <= 12 * lr and np.mean(diff > 1e-3 * lr) <= 0.05, (diff.max(), np.mean(diff > 1e-3 * lr))
    a.close()
    b.close()
