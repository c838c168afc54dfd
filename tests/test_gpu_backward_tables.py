"""The adjoint at the scene sizes where its shared memory needs the opt-in: 100 bytes per object and 12 per endpoint of
tables and sums, 4160 bytes of queue, 48 KB without the opt-in.  A scene padded to such a size with objects that no
sequence uses has the gradients of the scene without them: the paths are the same bit for bit, so the sums agree up to the
order of their additions (FP32 partial sums, FP64 totals: 1e-5 of the largest entry), and the padding gets zero.  The opt-in lasts
for the process, so the sizes run in one of their own, smallest first."""
import subprocess
import sys

import numpy as np
import pytest

import conftest  # noqa: F401  (run as a program: the repository on the path)
from paper_2510_16172_gb300 import fpt, scenes

pytestmark = pytest.mark.gpu

# one TX, one RX: 449 objects are the last without the opt-in, 491 the last whose dynamic part is below 48 KB by itself
USED, SIZES = 440, (448, 449, 450, 455, 491, 492)


def gradients(ctx, n_obj):
    import torch

    sc = scenes.city(2, n_obj=USED, n_rx=1)
    more = np.arange(n_obj) % USED  # copies of the first objects behind them
    put = lambda a: torch.as_tensor(a, dtype=torch.float32, device="cuda")  # noqa: E731
    # (on the device, where the centre is given: the host upload takes it from the vertices)
    scene = fpt.Scene(ctx, sc.types[more], put(sc.verts[more]), put(sc.tx), put(sc.rx), centre=np.array([250.0, 250.0, 30.0]))
    batch = fpt.Batch.seeded(ctx, scene, 5, 3000, 1, 5, np.arange(USED, dtype=np.int32))
    out = fpt.solve(ctx, scene, batch)
    dX, dL = (put(a) for a in scenes.cotangents(7, batch.n_paths, 5))
    sums = [fpt.backward(ctx, scene, batch, out["T"], out["status"], dX, dL),
            fpt.backward_noalloc(ctx, scene, batch, out["T"], out["status"], dX, dL),
            fpt.solve_grad(ctx, scene, batch, dX=dX, dL=dL)[1]]
    ctx.sync()
    return out["T"].clone(), out["status"].clone(), [[g.clone() for g in s] for s in sums]


def check():
    import torch

    ctx = fpt.Context(0)
    T0, st0, sums0 = gradients(ctx, USED)
    assert int(((st0 & fpt.ST_SOLVED) > 0).sum()) > 1000
    for n_obj in SIZES:
        T, st, sums = gradients(ctx, n_obj)
        assert torch.equal(T, T0) and torch.equal(st, st0), n_obj
        for s, s0 in zip(sums, sums0):
            for g, want in zip(s, s0):
                assert bool((g[len(want):] == 0).all()), n_obj
                assert float((g[:len(want)] - want).abs().max()) <= 1e-5 * float(want.abs().max()), n_obj


def test_backward_around_the_opt_in():
    from paper_2510_16172_gb300 import build

    build.build()
    r = subprocess.run([sys.executable, __file__], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    check()
