"""Orders of one call side by side against the same orders one after the other.

A call whose batch holds several orders runs them on streams of their own, each with its own scratch
and counters; with kernel timing on (and for large batches) it runs them in sequence on the context's
stream.  Paths are independent, so both ways give the same outputs bit for bit; the gradient sums agree up
to the order of additions (FP32 partial sums of at most 64 tiles, FP64 totals: 1e-5 of the largest entry).
"""

import pytest

import oracle
from paper_2510_16172_gb300 import fpt, scenes

pytestmark = pytest.mark.gpu

MASK = fpt.ST_VALID | fpt.ST_SOLVED


@pytest.fixture(scope="module")
def ctx():
    import torch

    from paper_2510_16172_gb300 import build

    build.build()
    oracle.build()
    assert torch.cuda.is_available()
    return fpt.Context(0)


def _batch(ctx, kind):
    import torch

    if kind == "canyon-1-3":  # one order far larger than the others
        sc = scenes.urban_canyon(0, rx_grid=3)
        scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
        return scene, fpt.Batch.exhaustive(ctx, scene, 1, 3, sc.alphabet)
    if kind == "pattern-launches":  # order 2 has pattern buckets of its own beside the unified launches
        sc = scenes.city(1, n_rx=4)
        scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
        return scene, fpt.Batch.seeded(ctx, scene, 3, 700_001, 1, 2)
    sc = scenes.tiny_scene(4, n_rx=2)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    if kind == "orders-1-10":  # more orders than streams
        return scene, fpt.Batch.seeded(ctx, scene, 9, 1500, 1, 10)
    # explicit, with an order that holds a single path and orders that hold none
    full = fpt.Batch.exhaustive(ctx, scene, 1, 2)
    ids, order, ti, ri = fpt.enumerate(ctx, full)
    wide = torch.full((len(order) + 1, 5), -1, dtype=torch.int32, device=ids.device)
    wide[:-1, :2] = ids
    wide[-1] = torch.tensor([0, 3, 9, 1, 4], dtype=torch.int32)
    one = lambda t, v: torch.cat([t, torch.tensor([v], dtype=t.dtype, device=t.device)])  # noqa: E731
    return scene, fpt.Batch.explicit(ctx, scene, wide, one(order, 5), one(ti, 0), one(ri, 1))


@pytest.mark.parametrize("kind", ["canyon-1-3", "pattern-launches", "orders-1-10", "explicit"])
def test_overlapped_orders_match_sequential_orders(ctx, kind):
    import torch

    scene, batch = _batch(ctx, kind)
    gen = torch.Generator(device="cuda").manual_seed(1)
    dX = torch.randn((batch.n_paths, batch.n_max, 3), generator=gen, device="cuda")

    def everything():
        out, grads = fpt.solve_grad(ctx, scene, batch, fpt.default_params(max_iters=32), dL_status_mask=MASK)
        again = fpt.solve(ctx, scene, batch, fpt.default_params(max_iters=32))
        ok = ((again["status"] & MASK) == MASK).float()
        bwd = fpt.backward(ctx, scene, batch, again["T"], again["status"], dX * ok[:, None, None], None)
        val = fpt.validity(ctx, scene, batch, again["T"])
        occ = fpt.occlusion(ctx, scene, batch, again["T"], again["status"], MASK)
        ctx.sync()
        exact = [*out.values(), *again.values(), *val, occ]
        return [t.clone() for t in exact], [t.clone() for t in (*grads, *bwd)]

    side, side_sums = everything()
    fpt.profile_enable(ctx, True)
    try:
        seq, seq_sums = everything()
    finally:
        fpt.profile_enable(ctx, False)
        fpt.profile_read(ctx)
    for a, b in zip(side, seq):
        assert torch.equal(torch.nan_to_num(a.float(), nan=7e30), torch.nan_to_num(b.float(), nan=7e30))
    for a, b in zip(side_sums, seq_sums):
        assert float((a - b).abs().max()) <= 1e-5 * max(1e-30, float(b.abs().max()))


def test_overlapped_unrolled_orders_match_sequential_orders(ctx):
    """Reverse mode through the steps: orders side by side (each with its own tape) against one after the other."""
    import torch

    scene, batch = _batch(ctx, "orders-1-10")

    def run():
        out = fpt.backward_unrolled(ctx, scene, batch, 5, 1, dL=torch.ones(batch.n_paths, device="cuda"), want_T=True)
        ctx.sync()
        return [t.clone() for t in out]

    side = run()
    fpt.profile_enable(ctx, True)
    try:
        seq = run()
    finally:
        fpt.profile_enable(ctx, False)
        fpt.profile_read(ctx)
    for k, (a, b) in enumerate(zip(side, seq)):
        if k < 3:
            assert float((a - b).abs().max()) <= 1e-5 * max(1e-30, float(b.abs().max()))
        else:
            assert torch.equal(torch.nan_to_num(a.float(), nan=7e30), torch.nan_to_num(b.float(), nan=7e30))
