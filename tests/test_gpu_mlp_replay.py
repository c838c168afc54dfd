"""Captured calls of the network: replayed after its parameters were set anew they use the new ones throughout, and a
forward pass no larger than a training batch before it needs no memory of its own (a capture cannot allocate)."""
import pytest

from paper_2510_16172_gb300 import fpt, scenes
from test_gpu_mlp import SCALE, numpy_params

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    from paper_2510_16172_gb300 import build

    build.build()
    return fpt.Context(0)


def capture(ctx, call):
    import torch

    old = ctx.stream
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.set_stream(torch.cuda.current_stream())
        out = call()
    ctx.set_stream(old)
    return g, out


def test_replayed_inference_uses_the_parameters_set_last(ctx):
    import torch

    sc = scenes.tiny_scene(51, n_rx=2)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    batch = fpt.Batch.seeded(ctx, scene, 9, 700, 1, 5)
    net = fpt.Mlp(ctx, 0, SCALE)
    net.set_params(numpy_params(1))
    first = net.infer(scene, batch).clone()
    g, T = capture(ctx, lambda: net.infer(scene, batch))
    net.set_params(numpy_params(2))
    g.replay()
    torch.cuda.synchronize()
    replayed = T.clone()
    want = net.infer(scene, batch)
    ctx.sync()
    assert torch.equal(replayed, want) and not torch.equal(first, want)
    net.close()


def test_replayed_training_step_uses_the_parameters_set_last(ctx):
    """A step moves a weight by at most about the learning rate, so one that starts from other layouts than the weights'
    own is far off in its gradient's signs: the same start gives the same step (up to the order of FP32 sums, which may turn
    the sign of a gradient that is zero but for rounding: 1 % of the weights)."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(4)
    X = (2.0 * torch.rand((1000, 64), generator=gen, device="cuda") - 1.0).to(torch.bfloat16)
    T = 2.0 * torch.rand((1000, 8), generator=gen, device="cuda") - 0.5
    G = torch.randn((1000, 12), generator=gen, device="cuda") ** 2
    lr = 1e-3
    a, b = fpt.Mlp(ctx, 0, SCALE), fpt.Mlp(ctx, 0, SCALE)
    a.set_params(numpy_params(1))
    a.train_step(X, T, G, lr)  # warm-up: workspace
    a.set_params(numpy_params(1))
    g, _ = capture(ctx, lambda: a.train_step(X, T, G, lr, want_loss=False))
    a.set_params(numpy_params(2))
    g.replay()
    torch.cuda.synchronize()
    b.set_params(numpy_params(2))
    b.train_step(X, T, G, lr)
    diff = abs(a.get_params() - b.get_params())
    assert (diff > 1e-3 * lr).mean() <= 0.01, (diff > 1e-3 * lr).mean()
    a.close()
    b.close()


@pytest.mark.parametrize("n", [1, 100, 1000])
def test_captured_forward_after_training_allocates_nothing(ctx, n):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(n)
    X = (2.0 * torch.rand((1000, 64), generator=gen, device="cuda") - 1.0).to(torch.bfloat16)
    T, G = torch.rand((1000, 8), generator=gen, device="cuda"), torch.rand((1000, 12), generator=gen, device="cuda")
    a, b = fpt.Mlp(ctx, 0, SCALE), fpt.Mlp(ctx, 0, SCALE)
    for net in (a, b):
        net.set_params(numpy_params(3))
    a.loss_grad(X, T, G)
    rows = X[:n].clone()
    g, Y = capture(ctx, lambda: a.forward(rows))
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, b.forward(rows))
    a.close()
    b.close()


def test_graphs_outlive_their_workspace(ctx):
    """A captured forward pass and a captured training step, replayed after larger ones of the same network; the step against
    one of a second network from the same parameters (see above)."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(8)
    X = (2.0 * torch.rand((20_000, 64), generator=gen, device="cuda") - 1.0).to(torch.bfloat16)
    T = 2.0 * torch.rand((20_000, 8), generator=gen, device="cuda") - 0.5
    G = torch.randn((20_000, 12), generator=gen, device="cuda") ** 2
    lr = 1e-3
    few = [t[:700].clone() for t in (X, T, G)]
    a, b = fpt.Mlp(ctx, 0, SCALE), fpt.Mlp(ctx, 0, SCALE)
    for net in (a, b):
        net.set_params(numpy_params(5))
    want = b.forward(few[0])
    a.loss_grad(*few)
    forward, Y = capture(ctx, lambda: a.forward(few[0]))
    step, _ = capture(ctx, lambda: a.train_step(*few, lr, want_loss=False))
    a.loss_grad(X, T, G)
    a.set_params(numpy_params(5))
    Y.zero_()
    forward.replay()
    step.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y, want)
    b.train_step(*few, lr)
    diff = abs(a.get_params() - b.get_params())
    assert (diff > 1e-3 * lr).mean() <= 0.01, (diff > 1e-3 * lr).mean()
    a.close()
    b.close()
