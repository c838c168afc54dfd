"""The training pass repeated on one batch while another stream keeps the memory busy: the same gradient every time.

A CTA pair's MMAs overwrite, layer by layer, the tensor-memory regions whose derivatives its epilogues read; an MMA that
does not wait for both CTAs' epilogues gives wrong layer gradients whenever one of them falls behind.  The
repeats differ only in the order of the FP32 additions: at most 76 partial sums per entry (one per pair for the biases,
28 batch slices for the weights), so by no more than 76 eps sum|partials|, eps = 2^-24; the partials are sums of independent
rows, so sum|partials| is about sqrt(76) times the entry's own scale: 4e-5 of a layer's largest entry, and 1e-4 is
allowed.  One warp's rows (32 of 8192) with wrong derivatives move an entry by about sqrt(32 / 8192) = 6 % of its scale.
"""
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


@pytest.mark.parametrize("n", [256, 8192, 30_001])
def test_repeated_gradients_agree(ctx, n):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(n)
    X = (2.0 * torch.rand((n, 64), generator=gen, device="cuda") - 1.0).to(torch.bfloat16)
    T = 2.0 * torch.rand((n, 8), generator=gen, device="cuda") - 0.5
    G = torch.randn((n, 12), generator=gen, device="cuda") ** 2
    net = fpt.Mlp(ctx, 0, SCALE)
    net.set_params(numpy_params(8))
    quiet_loss, quiet = net.loss_grad(X, T, G)
    quiet = quiet.clone()
    busy = torch.cuda.Stream()
    a = torch.zeros(1 << 27, device="cuda")
    b = torch.empty_like(a)
    torch.cuda.synchronize()
    runs = []
    for _ in range(24):
        with torch.cuda.stream(busy):
            b.copy_(a)
        loss, g = net.loss_grad(X, T, G)
        assert abs(loss - quiet_loss) <= 1e-4 * abs(quiet_loss)
        runs.append(g.clone())
    torch.cuda.synchronize()
    at = 0
    for name, shape in mo.SIZES:
        layer = slice(at, at + int(np.prod(shape)))
        at = layer.stop
        bound = 1e-4 * float(quiet[layer].abs().max())
        for g in runs:
            assert float((g[layer] - quiet[layer]).abs().max()) <= bound, name
    net.close()


def test_train_refuses_a_learning_rate_decayed_to_zero(ctx):
    """As fpt_mlp_train_step refuses it: 1e-3, 1e-23, 1e-43 (subnormal), then zero in FP32."""
    import torch

    net = fpt.Mlp(ctx, 5, SCALE)
    X = torch.zeros((128, 64), dtype=torch.bfloat16, device="cuda")
    T, G = torch.zeros((128, 8), device="cuda"), torch.zeros((128, 12), device="cuda")
    assert len(net.train(X, T, G, epochs=3, batch=128, lr=1e-3, lr_decay=1e-20)) == 3
    with pytest.raises(fpt.FptError, match="learning rate"):
        net.train(X, T, G, epochs=4, batch=128, lr=1e-3, lr_decay=1e-20)
    with pytest.raises(fpt.FptError, match="learning rate"):
        net.train_step(X, T, G, 0.0)
    net.close()


def permutation(n, seed, epoch):
    """The samples of an epoch in their order: the seeded Feistel permutation of [0, n), in whole-array form."""
    u = np.uint64
    gold = 0x9E3779B97F4A7C15

    def mix(z):
        z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
        return z ^ (z >> u(31))

    h = 1
    while 4 ** h < n:
        h += 1
    mask = u((1 << h) - 1)
    with np.errstate(over="ignore"):
        key = mix(np.array([(seed + gold * (epoch + 2)) % 2 ** 64], dtype=u))[0]
        x = np.arange(n, dtype=u)
        todo = np.ones(n, dtype=bool)
        while todo.any():
            left, right = x[todo] >> u(h), x[todo] & mask
            for k in range(4):
                f = mix(right ^ (key + u(gold * (k + 1) % 2 ** 64))) & mask
                left, right = right, left ^ f
            x[todo] = (left << u(h)) | right
            todo = x >= n
    return x.astype(np.int64)


def test_chained_steps_on_shuffled_batches(ctx):
    """Two epochs of two steps in one call, batches of more than one tile per pair with ragged last tiles and rows left over,
    against single steps on rows gathered here by the same permutation.  The same gradients up to the order of FP32 sums: the
    weights agree to 1e-3 lr but for those whose gradient is zero but for rounding (as in the test of whole-set batches),
    and fewer than one in a thousand take a step the other way."""
    import torch

    n, batch, lr = 21_001, 10_113, 1e-3
    order = permutation(n, 3, 0)
    assert np.array_equal(np.sort(order), np.arange(n))
    gen = torch.Generator(device="cuda").manual_seed(6)
    X = (2.0 * torch.rand((n, 64), generator=gen, device="cuda") - 1.0).to(torch.bfloat16)
    T = 2.0 * torch.rand((n, 8), generator=gen, device="cuda") - 0.5
    G = torch.randn((n, 12), generator=gen, device="cuda") ** 2
    a, b = fpt.Mlp(ctx, 7, SCALE), fpt.Mlp(ctx, 7, SCALE)
    hist = a.train(X, T, G, epochs=2, batch=batch, lr=lr, lr_decay=0.5, seed=3)
    losses = []
    for epoch in range(2):
        order = torch.as_tensor(permutation(n, 3, epoch), device="cuda")
        for k in range(2):
            rows = order[k * batch:(k + 1) * batch]
            losses.append(b.train_step(X[rows].contiguous(), T[rows].contiguous(), G[rows].contiguous(), lr * 0.5 ** epoch))
    np.testing.assert_allclose(hist, np.reshape(losses, (2, 2)).mean(axis=1), rtol=1e-4)
    diff = np.abs(a.get_params() - b.get_params())
    assert np.mean(diff > 1e-3 * lr) <= 0.05 and np.quantile(diff, 0.999) <= lr, np.quantile(diff, [0.9, 0.99, 0.999, 1.0])
    a.close()
    b.close()
