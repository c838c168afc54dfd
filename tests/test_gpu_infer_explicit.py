"""The learned start of an explicit batch with unusable sequences among the others: every slot of the output is written."""
import numpy as np
import pytest

from paper_2510_16172_gb300 import fpt, scenes
from test_gpu_mlp import SCALE, numpy_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_max", [3, 7])
def test_every_slot_of_an_explicit_batch_is_written(n_max):
    """Sequences of orders 1..n_max, then the same with an object, endpoint or order out of range.  The good ones get what they
    get in a batch of their own bit for bit (each path is one row of the network); the others start at 1/2 in the
    slots of their order (clipped to 1..n_max); slots past the order are zero."""
    import torch

    from paper_2510_16172_gb300 import build

    build.build()
    ctx = fpt.Context(0)
    sc = scenes.tiny_scene(51, n_rx=2)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    rng = np.random.default_rng(n_max)
    n = 300
    order = rng.integers(1, n_max + 1, n)
    ids = np.cumsum(rng.integers(1, sc.n_obj, (n, n_max)), axis=1) % sc.n_obj
    ti, ri = np.zeros(n, dtype=int), rng.integers(0, 2, n)
    bad = rng.random(n) < 0.4
    kind = rng.integers(0, 4, n)
    ids2, order2, ti2, ri2 = ids.copy(), order.copy(), ti.copy(), ri.copy()
    ids2[bad & (kind == 0), 0] = sc.n_obj
    order2[bad & (kind == 1)] = 0
    order2[bad & (kind == 2)] = n_max + 1
    ri2[bad & (kind == 3)] = 2

    def put(a, dtype):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")

    def infer(net, ids, order, ti, ri):
        batch = fpt.Batch.explicit(ctx, scene, put(ids, torch.int32), put(order, torch.uint8), put(ti, torch.int32),
                                   put(ri, torch.int32))
        T = torch.full((n, n_max, 2), float("nan"), device="cuda")
        net.infer(scene, batch, out=T)
        ctx.sync()
        return T.cpu().numpy()

    net = fpt.Mlp(ctx, 0, SCALE)
    net.set_params(numpy_params(51))
    good, T = infer(net, ids, order, ti, ri), infer(net, ids2, order2, ti2, ri2)
    net.close()
    assert np.isfinite(T).all() and np.array_equal(T[~bad], good[~bad])
    slots = np.arange(n_max)[None, :, None] < np.clip(order2, 1, n_max)[:, None, None]
    assert np.array_equal(T[bad], np.broadcast_to(np.where(slots, 0.5, 0.0), T.shape)[bad])
    assert (good[~np.broadcast_to(np.arange(n_max)[None, :, None] < order[:, None, None], good.shape)] == 0).all()
