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
