"""Calls captured into CUDA graphs and the context's scratch.

A captured call takes the scratch as it stands: where an earlier call left only the largest order's (kernel timing runs the
orders in turn), the captured one runs them in turn too.  And a graph stays usable after later calls outgrow the scratch
it was captured with.  Paths are independent: the replayed outputs are those of a direct call bit for bit, the gradient sums up
to the order of additions (FP32 partial sums, FP64 totals: 1e-5 of the largest entry)."""
import pytest

from paper_2510_16172_gb300 import fpt, scenes

pytestmark = pytest.mark.gpu

MASK = fpt.ST_VALID | fpt.ST_SOLVED


@pytest.fixture()
def ctx():
    from paper_2510_16172_gb300 import build

    build.build()
    return fpt.Context(0)


def batch_of(ctx, per_pair, lo=1, hi=4):
    sc = scenes.tiny_scene(2, n_rx=2)
    scene = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    return scene, fpt.Batch.seeded(ctx, scene, 17, per_pair, lo, hi)


def everything(ctx, scene, batch):
    """Outputs that must agree bit for bit, and sums."""
    import torch

    out, grads = fpt.solve_grad(ctx, scene, batch, dL_status_mask=MASK)
    mask, bdist, _ = fpt.validity(ctx, scene, batch, out["T"])
    occ = fpt.occlusion(ctx, scene, batch, out["T"], out["status"], MASK)
    bwd = fpt.backward(ctx, scene, batch, out["T"], out["status"], None, torch.ones(batch.n_paths, device="cuda"))
    unrolled = fpt.backward_unrolled(ctx, scene, batch, 3, 1, dL=torch.ones(batch.n_paths, device="cuda"), want_T=True)
    return [out["T"], out["status"], out["L"], mask, bdist, occ, *unrolled[3:]], [*grads, *bwd, *unrolled[:3]]


def agree(got, want):
    import torch

    for a, b in zip(got[0], want[0]):
        assert torch.equal(torch.nan_to_num(a.float(), nan=7e30), torch.nan_to_num(b.float(), nan=7e30))
    for a, b in zip(got[1], want[1]):
        assert float((a - b).abs().max()) <= 1e-5 * max(1e-30, float(b.abs().max()))


def captured(ctx, scene, batch):
    import torch

    old = ctx.stream
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ctx.set_stream(torch.cuda.current_stream())
        out = everything(ctx, scene, batch)
    ctx.set_stream(old)
    return g, out


def replayed(g, out):
    import torch

    for t in [*out[0], *out[1]]:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    return out


def test_capture_with_the_scratch_of_orders_in_turn(ctx):
    scene, batch = batch_of(ctx, 3000)
    fpt.profile_enable(ctx, True)
    want = everything(ctx, scene, batch)
    ctx.sync()
    fpt.profile_enable(ctx, False)
    fpt.profile_read(ctx)
    g, out = captured(ctx, scene, batch)
    agree(replayed(g, out), want)


def test_graph_outlives_its_scratch(ctx):
    import torch

    scene, batch = batch_of(ctx, 3000)
    want = everything(ctx, scene, batch)
    ctx.sync()
    g, out = captured(ctx, scene, batch)
    agree(replayed(g, out), want)
    large = batch_of(ctx, 60_000, 1, 6)
    direct = everything(ctx, *large)
    ctx.sync()
    agree(replayed(g, out), want)
    again = everything(ctx, *large)
    torch.cuda.synchronize()
    agree(again, direct)


def test_graph_outlives_its_accumulators(ctx):
    """The gradient sums are sized for the scene: a later call on a larger one."""
    scene, batch = batch_of(ctx, 3000)
    want = everything(ctx, scene, batch)
    ctx.sync()
    g, out = captured(ctx, scene, batch)
    sc = scenes.city(1, n_obj=400, n_rx=2)
    other = fpt.Scene(ctx, sc.types, sc.verts, sc.tx, sc.rx)
    small = fpt.Batch.seeded(ctx, other, 17, 1000, 1, 4)
    direct = everything(ctx, other, small)
    ctx.sync()
    agree(replayed(g, out), want)
    agree(everything(ctx, other, small), direct)
