"""Point cotangents on few paths: the adjoint's queue against a batch of only those paths."""

import pytest

import oracle
from paper_2510_16172_gb300 import fpt, scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2510_16172_gb300 import build

    build.build()
    oracle.build()
    return fpt.Context(0)


@pytest.mark.parametrize("count,rx_grid", [(0, 1), (1, 1), (127, 2), (128, 2), (129, 2), (5000, 4), (None, 2)])
def test_sparse_cotangents_match_their_own_batch(ctx, count, rx_grid):
    """`count` paths of a canyon (None: every path that takes part) carry dX; the explicit batch holds them alone.  Equal up
    to the order of the sums (FP32 partial sums, FP64 totals)."""
    import torch

    sc = scenes.urban_canyon(3, rx_grid=rx_grid)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    batch = fpt.Batch.exhaustive(ctx, scene, 1, 3, sc.alphabet)
    out = fpt.solve(ctx, scene, batch)
    ok = torch.nonzero((out["status"] & (fpt.ST_VALID | fpt.ST_SOLVED)) == (fpt.ST_VALID | fpt.ST_SOLVED)).squeeze(1)
    gen = torch.Generator(device="cuda").manual_seed(1)
    pick = ok if count is None else ok[torch.randperm(len(ok), generator=gen, device="cuda")[:count]].sort().values
    assert count is None or len(pick) == count
    dX = torch.zeros((batch.n_paths, batch.n_max, 3), device="cuda")
    dX[pick] = torch.randn((len(pick), batch.n_max, 3), generator=gen, device="cuda")
    got = fpt.backward(ctx, scene, batch, out["T"], out["status"], dX, None)
    ids, order, ti, ri = fpt.enumerate(ctx, batch)
    alone = fpt.Batch.explicit(ctx, scene, ids[pick].contiguous(), order[pick].contiguous(), ti[pick].contiguous(),
                               ri[pick].contiguous())
    want = fpt.backward(ctx, scene, alone, out["T"][pick].contiguous(), out["status"][pick].contiguous(),
                        dX[pick].contiguous(), None)
    ctx.sync()
    for a, b in zip(got, want):
        assert float((a - b).abs().max()) <= 1e-5 * float(b.abs().max())
