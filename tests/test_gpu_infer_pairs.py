"""Fused inference on CTA pairs: sizes at the edges of its tiles (128 paths per CTA, 256 per pair and step, several
steps per pair), against the FP64 forward pass of the network."""
import numpy as np
import pytest

import oracle
from oracle import mlp_oracle as mo
from paper_2510_16172_gb300 import fpt, scenes
from test_gpu_mlp import SCALE, numpy_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2510_16172_gb300 import build

    build.build()
    oracle.build()
    return fpt.Context(0)


@pytest.mark.parametrize("per_pair,n_rx,lo,hi", [(1, 1, 1, 1), (128, 1, 1, 4), (129, 1, 2, 5), (257, 1, 1, 5),
                                                 (20_001, 3, 1, 5), (20_003, 2, 4, 7)])
def test_infer_tile_edges(ctx, per_pair, n_rx, lo, hi):
    sc = scenes.tiny_scene(51, n_rx=n_rx)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    batch = fpt.Batch.seeded(ctx, scene, 9, per_pair, lo, hi)
    params = numpy_params(51)
    net = fpt.Mlp(ctx, 0, SCALE)
    net.set_params(params)
    T = net.infer(scene, batch)
    ctx.sync()
    T = T.cpu().numpy()
    net.close()
    ids, order, ti, ri = oracle.seeded_paths(sc, 9, per_pair, lo, hi)
    F, _ = mo.features(sc, ids, order, ti, ri, SCALE)
    Y = mo.forward(params.astype(np.float64), mo.bf16(F))["Y"]
    expect = np.zeros(T.shape)
    for p in range(len(order)):
        expect[p, :order[p]] = 0.5
        for s in range(min(order[p], 4)):
            expect[p, s, 0] = Y[p, 2 * s]
            if sc.types[ids[p, s]] == scenes.QUAD:
                expect[p, s, 1] = Y[p, 2 * s + 1]
    # the bound of the other fused-inference tests: BF16 activations and weights through four layers
    assert np.abs(T - expect).max() <= 5e-3 * max(1.0, np.abs(Y).max())
    unused = np.arange(T.shape[1])[None, :] >= order[:, None]
    assert (T[unused] == 0).all()
