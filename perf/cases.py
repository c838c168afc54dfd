"""The work that users of the library have it do, as cases that can be timed and compared.

Every case goes through the Python API (``fpt``, ``autograd``): a differentiable solve of a tiny scene,
solves of exhaustive and seeded batches from thousands to tens of millions of paths with their implicit
gradients, the single parts that programs call by themselves (backward with point cotangents, validity,
obstruction, reverse mode through the iterations, the network's prediction) and a training run of the
network.  Scenes come from the package's seeded generators with the sizes of its benchmark and tests.

``exact`` gives 64-bit values for the parts that have them.  A solve has none as a whole: the iterate of
a path that ends unsolved (a kinked minimiser, the step cap) is a value of the FP32 iteration itself, and
which paths enter the gradient sums depends on it.
"""

import math

import numpy as np
import torch

from paper_2510_16172_gb300 import fpt, scenes
from paper_2510_16172_gb300.autograd import FermatSolver

VALID_SOLVED = fpt.ST_VALID | fpt.ST_SOLVED
NO_GRADIENT = fpt.ST_REPEAT | fpt.ST_INVALID_INPUT | fpt.ST_DEGENERATE | fpt.ST_NONFINITE


def listed():
    return [
        # a differentiable solve and its backward in an optimisation loop over a small scene: the smallest
        # call, one TX and RX, all 156 sequences of order 1-2 over 12 objects, geometry on the GPU
        {"name": "autograd_tiny", "kind": "autograd", "quads": 8, "edges": 4, "n_rx": 1, "hi": 2},
        # evaluating starts on one random 10 m scene: seeded sequences of order 1-4, step cap 32
        {"name": "tiny_seeded", "kind": "solve_tiny", "paths": 200_000, "lo": 1, "hi": 4, "max_iters": 32},
        # an urban canyon with a few receivers, every sequence of order 1-3, the library's default settings
        {"name": "canyon_sector", "kind": "solve_canyon", "rx_grid": 4, "lo": 1, "hi": 3, "max_iters": 64},
        # the benchmark's urban canyon: 33.5 M paths of order 3, step cap 32
        {"name": "canyon_full", "kind": "solve_canyon", "rx_grid": 32, "lo": 3, "hi": 3, "max_iters": 32},
        # a ragged city batch: seeded sequences of order 1-5 over 256 objects, 16 receivers, an odd count
        {"name": "city_ragged", "kind": "solve_city", "per_pair": 500_003, "hi": 5, "max_iters": 32},
        # long sequences (the inverse Hessian in shared memory), orders 6-8
        {"name": "long_orders", "kind": "solve_tiny", "paths": 100_000, "lo": 6, "hi": 8, "max_iters": 64},
        # the backward of a loss on the points and lengths of the valid paths (what autograd passes on)
        {"name": "points_backward", "kind": "backward", "rx_grid": 8, "lo": 1, "hi": 3},
        # validity, boundary distance and residual of given parameters, city sequences of order 1-5
        {"name": "validity_city", "kind": "validity", "per_pair": 62_501, "hi": 5},
        # which segments of the valid solved canyon paths are obstructed
        {"name": "occlusion_canyon", "kind": "occlusion", "rx_grid": 16, "lo": 3, "hi": 3},
        # the gradient through 16 solver steps (the comparison with the implicit gradient), orders 1-3
        {"name": "unrolled_16", "kind": "unrolled", "paths": 300_000, "lo": 1, "hi": 3, "steps": 16, "rounds": 1},
        # the network's starting parameters for a city batch of orders 1-5
        {"name": "infer_city", "kind": "infer", "per_pair": 250_001, "hi": 5},
        # one epoch of Adam over half a million samples at the training loop's default batch
        {"name": "train_8192", "kind": "train", "samples": 524_288, "batch": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["autograd", "solve_tiny", "solve_canyon", "solve_canyon", "solve_city", "solve_city",
                       "solve_long", "backward", "validity", "occlusion", "unrolled", "infer", "train"])
    if kind == "autograd":
        return {"kind": kind, "quads": rng.randint(4, 10), "edges": rng.randint(2, 7), "n_rx": rng.randint(1, 9),
                "hi": rng.randint(1, 3)}
    if kind == "solve_tiny":
        lo = rng.randint(1, 2)
        return {"kind": kind, "paths": _log_int(rng, 1000, 2_000_000), "lo": lo, "hi": rng.randint(lo, 5),
                "max_iters": rng.choice([32, 64])}
    if kind == "solve_long":
        lo = rng.randint(5, 9)
        return {"kind": "solve_tiny", "paths": _log_int(rng, 1000, 200_000), "lo": lo, "hi": rng.randint(max(lo, 6), 10),
                "max_iters": 64}
    if kind == "solve_canyon":
        lo = rng.randint(1, 3)
        return {"kind": kind, "rx_grid": _log_int(rng, 1, 24), "lo": lo, "hi": 3, "max_iters": rng.choice([32, 64])}
    if kind == "solve_city":
        return {"kind": kind, "per_pair": _log_int(rng, 500, 600_000), "hi": rng.randint(2, 5),
                "max_iters": rng.choice([32, 64])}
    if kind == "backward":
        return {"kind": kind, "rx_grid": rng.randint(1, 11), "lo": rng.randint(1, 3), "hi": 3}
    if kind == "validity":
        return {"kind": kind, "per_pair": _log_int(rng, 300, 125_000), "hi": rng.randint(1, 5)}
    if kind == "occlusion":
        return {"kind": kind, "rx_grid": rng.randint(2, 24), "lo": rng.randint(1, 3), "hi": 3}
    if kind == "unrolled":
        lo = rng.randint(1, 3)
        return {"kind": kind, "paths": _log_int(rng, 1000, 500_000), "lo": lo, "hi": rng.randint(lo, 4),
                "steps": rng.randint(4, 16), "rounds": rng.choice([1, 4])}
    if kind == "infer":
        return {"kind": kind, "per_pair": _log_int(rng, 500, 400_000), "hi": rng.randint(1, 6)}
    batch = rng.choice([2048, 4096, 8192, 16384, 65536])
    return {"kind": kind, "samples": batch * rng.randint(4, 8) + rng.randint(0, batch - 1), "batch": batch}


def _host_scene(case, seed):
    kind = case["kind"]
    if kind == "autograd":
        return scenes.tiny_scene(seed, case["quads"], case["edges"], 1, case["n_rx"])
    if kind in ("solve_tiny", "unrolled", "train"):
        return scenes.tiny_scene(seed)
    if kind in ("solve_canyon", "backward", "occlusion"):
        return scenes.urban_canyon(seed, rx_grid=case["rx_grid"])
    return scenes.city(seed)


def _scene(ctx, h):
    return fpt.Scene(ctx, h.types, h.verts, h.tx, h.rx)


def _batch(ctx, scene, h, case, seed):
    kind = case["kind"]
    if kind in ("solve_canyon", "backward", "occlusion"):
        return fpt.Batch.exhaustive(ctx, scene, case["lo"], case["hi"], h.alphabet)
    if "per_pair" in case:
        return fpt.Batch.seeded(ctx, scene, seed, case["per_pair"], 1, case["hi"])
    if kind == "train":  # enough sequences of order 1-4 that half of them give the samples
        return fpt.Batch.seeded(ctx, scene, seed, 2 * case["samples"], 1, 4)
    return fpt.Batch.seeded(ctx, scene, seed, case["paths"], case["lo"], case["hi"])


def _network(ctx, seed):
    return fpt.Mlp(ctx, seed, 10.0)


def _params(case):
    # step cap and kink stop of the benchmark at cap 32, the library's defaults otherwise
    kink = 0.01 if case["kind"] == "solve_canyon" and case["max_iters"] == 32 else 0.0
    return fpt.default_params(max_iters=case["max_iters"], kink_stop=kink)


def prepare(case, seed):
    h = _host_scene(case, seed)
    kind = case["kind"]
    if kind == "autograd":
        solver = FermatSolver(h.types, order_lo=1, order_hi=case["hi"], centre=h.verts.reshape(-1, 3).mean(axis=0))
        dev = solver.device
        geo = [torch.tensor(a, dtype=torch.float32, device=dev).requires_grad_(True) for a in (h.tx, h.rx, h.verts)]
        g = torch.Generator(device=dev).manual_seed(seed)
        n_pairs = len(h.tx) * len(h.rx)
        n = n_pairs * sum(h.n_obj ** k for k in range(1, case["hi"] + 1))
        w = torch.randn((n, case["hi"], 3), generator=g, device=dev)
        return {"case": case, "solver": solver, "geo": geo, "w": w}
    ctx = fpt.Context(0)
    scene = _scene(ctx, h)
    batch = _batch(ctx, scene, h, case, seed)
    s = {"case": case, "ctx": ctx, "scene": scene, "batch": batch, "host": h}
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev).manual_seed(seed)
    if kind.startswith("solve"):
        s["params"] = _params(case)
        s["out"] = fpt.alloc_outputs(ctx, batch, with_X=False, with_rho=False)
    elif kind == "backward":
        out = fpt.solve(ctx, scene, batch)
        keep = ((out["status"] & VALID_SOLVED) == VALID_SOLVED).float()
        s["T"], s["status"] = out["T"], out["status"]
        s["dX"] = torch.randn((batch.n_paths, batch.n_max, 3), generator=g, device=dev) * keep[:, None, None]
        s["dL"] = torch.randn(batch.n_paths, generator=g, device=dev) * keep
    elif kind in ("validity", "occlusion"):
        out = fpt.solve(ctx, scene, batch, out=fpt.alloc_outputs(ctx, batch, with_X=False, with_rho=False))
        s["T"], s["status"] = out["T"], out["status"]
    elif kind == "unrolled":
        s["dL"] = torch.ones(batch.n_paths, device=dev)
    elif kind == "infer":
        s["net"] = _network(ctx, seed)
    elif kind == "train":
        s["net"] = _network(ctx, seed)
        s["data"] = _dataset(s, g, case["samples"])
    return s


def _dataset(s, g, n):
    """Features, targets and Gram matrices of the solver's own solutions on one random scene, n samples."""
    ctx, scene, net = s["ctx"], s["scene"], s["net"]
    batch = s["batch"]
    out = fpt.solve(ctx, scene, batch, out=fpt.alloc_outputs(ctx, batch, with_X=False, with_rho=False))
    X, G = net.features(scene, batch, with_gram=True)
    idx = torch.nonzero((out["status"] & fpt.ST_SOLVED) > 0).squeeze(1)
    idx = idx[torch.arange(n, device=idx.device) % idx.numel()]
    T = out["T"].reshape(batch.n_paths, -1)[idx].contiguous()
    return X[idx].contiguous(), T, G[idx].contiguous()


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "autograd":
        tx, rx, verts = s["geo"]
        X, L, status = s["solver"](tx, rx, verts)
        keep = ((status & VALID_SOLVED) == VALID_SOLVED).float()
        loss = (L * keep).sum() + ((X * s["w"]).sum(dim=(1, 2)) * keep).sum()
        g_tx, g_rx, g_v = torch.autograd.grad(loss, (tx, rx, verts))
        return {"X": X.detach(), "L": L.detach(), "status": status, "g_tx": g_tx, "g_rx": g_rx, "g_verts": g_v}
    if kind.startswith("solve"):
        out, grads = fpt.solve_grad(s["ctx"], s["scene"], s["batch"], s["params"], dL_status_mask=VALID_SOLVED,
                                    out=s["out"])
        return {"T": out["T"], "L": out["L"], "status": out["status"], "iters": out["iters"], "grads": list(grads)}
    if kind == "backward":
        return list(fpt.backward(s["ctx"], s["scene"], s["batch"], s["T"], s["status"], s["dX"], s["dL"]))
    if kind == "validity":
        return list(fpt.validity(s["ctx"], s["scene"], s["batch"], s["T"]))
    if kind == "occlusion":
        return fpt.occlusion(s["ctx"], s["scene"], s["batch"], s["T"], s["status"], VALID_SOLVED)
    if kind == "unrolled":
        return list(fpt.backward_unrolled(s["ctx"], s["scene"], s["batch"], case["steps"], case["rounds"], dL=s["dL"],
                                          want_T=True))
    if kind == "infer":
        return s["net"].infer(s["scene"], s["batch"])
    X, T, G = s["data"]
    loss = s["net"].train(X, T, G, 1, batch=case["batch"])
    return {"loss": loss, "params": s["net"].get_params()}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _paths(case):
    """{order: number of paths} of a case."""
    kind = case["kind"]
    if kind == "autograd":
        K = case["quads"] + case["edges"]
        return {n: case["n_rx"] * K**n for n in range(1, case["hi"] + 1)}
    if kind in ("solve_canyon", "backward", "occlusion"):
        return {n: case["rx_grid"] ** 2 * 32**n for n in range(case["lo"], case["hi"] + 1)}
    lo = case.get("lo", 1)
    total = 16 * case["per_pair"] if "per_pair" in case else case["paths"]
    m = case["hi"] - lo + 1
    return {n: total / m for n in range(lo, case["hi"] + 1)}


def _step_flops(n, d=1.6):
    """FP32 operations of one BFGS step with one Eq. 6 round: n interactions, d unknowns each on average."""
    m = d * n
    grad = n * (6 * d) + (n + 1) * 17 + n * (3 + 5 * d)
    update = 2 * m * m + 4 * m * m + 2 * m * m + 12 * m
    search = n * 6 * d + (n + 1) * (3 + 10 + 12)
    return grad + update + search


MEAN_STEPS = 15.0  # BFGS steps to the step tolerance (measured means on canyon and city: 15-17)


def work(case):
    kind = case["kind"]
    if kind == "train":
        steps = case["samples"] // case["batch"]
        rows = steps * case["batch"]
        w = 64 * 256 + 2 * 256 * 256 + 256 * 16
        return {"bytes": rows * (128 + 32 + 48) + steps * 152336 * 4 * 6, "flops": rows * 6 * w}
    per = _paths(case)
    n_all = sum(per.values())
    n_max = case["hi"]
    t_bytes = 8 * n_max
    if kind == "infer":
        w = 64 * 256 + 2 * 256 * 256 + 256 * 16
        return {"bytes": n_all * t_bytes, "flops": n_all * 2 * w}
    if kind == "autograd":
        flops = sum(c * (MEAN_STEPS * _step_flops(n) + 600 * n) for n, c in per.items())
        return {"bytes": n_all * (t_bytes + 2 * 12 * n_max + 9), "flops": flops}
    if kind.startswith("solve"):
        flops = sum(c * (MEAN_STEPS * _step_flops(n) + 500 * n) for n, c in per.items())
        return {"bytes": n_all * (t_bytes + 6), "flops": flops}
    if kind == "backward":
        # the cotangents and statuses of every path, the parameters and arithmetic of the valid ones (7 %)
        return {"bytes": n_all * (12 * n_max + 4 + 1) + 0.07 * n_all * t_bytes,
                "flops": sum(0.07 * c * 200 * n for n, c in per.items())}
    if kind == "validity":
        return {"bytes": n_all * (t_bytes + 9), "flops": sum(c * 500 * n for n, c in per.items())}
    if kind == "occlusion":
        # the valid solved paths (7 %) against the 32 facades, one plane test per segment and facade
        return {"bytes": n_all * 3 + 0.07 * n_all * t_bytes,
                "flops": sum(0.07 * c * (n + 1) * 32 * 14 for n, c in per.items())}
    # unrolled: the forward's steps, and their reverse at about three times the forward's operations
    return {"bytes": n_all * (t_bytes + 5), "flops": sum(c * case["steps"] * 4 * _step_flops(n, 2.0) for n, c in per.items())}


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------
def _decoded(s):
    ids, order, ti, ri = fpt.enumerate(s["ctx"], s["batch"])
    return ids.long(), order.long(), ti.long(), ri.long()


def _geometry(h, dev):
    """b [K, 3], A [K, 2, 3], is_edge [K], TX, RX in 64 bits."""
    v = torch.tensor(h.verts, dtype=torch.float64, device=dev)
    edge = torch.tensor(h.types.astype(np.int64), device=dev) == scenes.EDGE
    A = torch.stack([v[:, 1] - v[:, 0], torch.where(edge[:, None], torch.zeros_like(v[:, 2]), v[:, 2] - v[:, 0])], 1)
    return (v[:, 0], A, edge, torch.tensor(h.tx, dtype=torch.float64, device=dev),
            torch.tensor(h.rx, dtype=torch.float64, device=dev))


def _points(b, A, T):
    return b + (A * T[..., None]).sum(-2)


def _grad_T(b, A, tx, rx, T):
    """grad_T L [P, n, 2] of paths with objects (b, A) [P, n, ...] (Eq. 5)."""
    x = torch.cat([tx[:, None], _points(b, A, T), rx[:, None]], 1)
    z = x[:, 1:] - x[:, :-1]
    u = z / z.norm(dim=-1, keepdim=True)
    return ((u[:, :-1] - u[:, 1:])[:, :, None] * A).sum(-1), u, z


def _hessian(b, A, edge, tx, rx, T):
    """The exact Hessian [P, 2n, 2n]; an edge's dead second parameter is decoupled."""
    n = T.shape[1]
    with torch.enable_grad():
        Tv = T.detach().requires_grad_(True)
        g = _grad_T(b.detach(), A.detach(), tx.detach(), rx.detach(), Tv)[0].reshape(-1, 2 * n)
        H = torch.stack([torch.autograd.grad(g[:, k].sum(), Tv, retain_graph=True)[0].reshape(-1, 2 * n)
                         for k in range(2 * n)], 1)
    i = torch.arange(n, device=T.device)
    own = H[:, 2 * i, 2 * i]
    H[:, 2 * i + 1, 2 * i + 1] = torch.where(edge, own, H[:, 2 * i + 1, 2 * i + 1])
    return H


def _exact_backward(s):
    h, dev = s["host"], s["T"].device
    ids, order, ti, ri = _decoded(s)
    v = torch.tensor(h.verts, dtype=torch.float64, device=dev)
    leaves = [torch.tensor(a, dtype=torch.float64, device=dev).requires_grad_(True) for a in (h.tx, h.rx)]
    v.requires_grad_(True)
    edge_k = torch.tensor(h.types.astype(np.int64), device=dev) == scenes.EDGE
    sums = [torch.zeros_like(t) for t in (*leaves, v)]
    use = ((s["status"] & NO_GRADIENT) == 0) & ((s["dL"] != 0) | (s["dX"] != 0).flatten(1).any(1))
    for n in range(1, s["batch"].n_max + 1):
        for p in torch.nonzero(use & (order == n)).squeeze(1).split(50_000):
            o = ids[p, :n]
            edge = edge_k[o]
            T = s["T"][p, :n].double()
            dX, dL = s["dX"][p, :n].double(), s["dL"][p].double()
            tx, rx, w = leaves[0][ti[p]], leaves[1][ri[p]], v[o]
            zero = torch.zeros_like(w[:, :, 2])
            A = torch.stack([w[:, :, 1] - w[:, :, 0], torch.where(edge[..., None], zero, w[:, :, 2] - w[:, :, 0])], 2)
            b = w[:, :, 0]
            g, _, z = _grad_T(b, A, tx, rx, T)
            vT = ((dX[:, :, None] * A).sum(-1) + dL[:, None, None] * g).detach().reshape(-1, 2 * n)
            lam = torch.linalg.solve(_hessian(b, A, edge, tx, rx, T), vT[..., None])[..., 0].reshape(-1, n, 2)
            # the explicit terms, less lam . d(grad_T L)/d(theta)
            total = (dX * _points(b, A, T)).sum() + (dL * z.norm(dim=-1).sum(-1)).sum() - (lam * g).sum()
            for t, d in zip(sums, torch.autograd.grad(total, (*leaves, v))):
                t += d
    return sums


def _exact_validity(s):
    h, dev = s["host"], s["T"].device
    b_k, A_k, edge_k, tx_k, rx_k = _geometry(h, dev)
    ids, order, ti, ri = _decoded(s)
    a0, a1 = A_k[:, 0], A_k[:, 1]
    n0 = a0.norm(dim=-1)
    # distance between the opposite sides: the area over the other side's length (an edge: its length)
    area = torch.linalg.cross(a0, a1).norm(dim=-1)
    h0 = torch.where(edge_k, n0, area / a1.norm(dim=-1).clamp_min(1e-300))
    h1 = area / n0
    N = s["batch"].n_paths
    bd = torch.empty(N, dtype=torch.float64, device=dev)
    for n in range(1, s["batch"].n_max + 1):
        p = torch.nonzero(order == n).squeeze(1)
        o = ids[p, :n]
        T = s["T"][p, :n].double()
        d = torch.minimum(T, 1 - T) * torch.stack([h0[o], h1[o]], -1)
        d[..., 1] = torch.where(edge_k[o], torch.full_like(d[..., 1], math.inf), d[..., 1])
        bd[p] = d.flatten(1).amin(1)
    return [None, bd, None]  # the mask is whole; the residual of a kinked path has no value


def _exact_infer(case, seed, s):
    h, dev = s["host"], torch.device("cuda", 0)
    p = torch.tensor(s["net"].get_params(), dtype=torch.float64, device=dev)
    sizes = [(256, 64), (256,), (256, 256), (256,), (256, 256), (256,), (16, 256), (16,)]
    layers, at = [], 0
    for z in sizes:
        layers.append(p[at:at + math.prod(z)].reshape(z))
        at += math.prod(z)
    b_k, A_k, edge_k, tx_k, rx_k = _geometry(h, dev)
    ids, order, ti, ri = _decoded(s)
    N, m = s["batch"].n_paths, s["batch"].n_max
    out = torch.zeros((N, m, 2), dtype=torch.float64, device=dev)
    S = 10.0
    for p0 in range(0, N, 400_000):
        q = slice(p0, min(N, p0 + 400_000))
        tx, rx, n = tx_k[ti[q]], rx_k[ri[q]], order[q]
        mid = 0.5 * (tx + rx)
        f = torch.zeros((len(n), 64), dtype=torch.float64, device=dev)
        f[:, 0:3], f[:, 3:6] = (tx - mid) / S, (rx - mid) / S
        for k in range(min(4, m)):
            o = ids[q, k].clamp_min(0)
            b, A, edge = b_k[o], A_k[o], edge_k[o]
            a1, a2 = A[:, 0], A[:, 1]
            g11, g12, g22 = (a1 * a1).sum(-1), (a1 * a2).sum(-1), (a2 * a2).sum(-1)
            det = torch.where(edge, torch.ones_like(g11), g11 * g22 - g12 * g12)
            tau, dist = [], []
            for pt in (tx, rx):
                r = pt - b
                c1, c2 = (a1 * r).sum(-1), (a2 * r).sum(-1)
                t1 = torch.where(edge, c1 / g11, (g22 * c1 - g12 * c2) / det)
                t2 = torch.where(edge, torch.zeros_like(c1), (g11 * c2 - g12 * c1) / det)
                tau.append(torch.stack([t1, t2], -1))
                dist.append((r - t1[:, None] * a1 - t2[:, None] * a2).norm(dim=-1) / S)
            ds = dist[0] + dist[1]
            w = torch.where((ds > 0)[:, None], (dist[1][:, None] * tau[0] + dist[0][:, None] * tau[1]) /
                            ds.clamp_min(1e-300)[:, None], 0.5 * (tau[0] + tau[1]))
            slot = torch.cat([torch.ones_like(ds)[:, None], edge.double()[:, None], tau[0], tau[1], dist[0][:, None],
                              dist[1][:, None], g11.sqrt()[:, None] / S, w], 1)
            f[:, 6 + 11 * k:17 + 11 * k] = torch.where((n > k)[:, None], slot, torch.zeros_like(slot))
        x = f
        for k in range(3):
            x = torch.nn.functional.gelu(x @ layers[2 * k].T + layers[2 * k + 1], approximate="tanh")
        y = (x @ layers[6].T + layers[7])[:, :8].reshape(-1, 4, 2)
        t = torch.full((len(n), m, 2), 0.5, dtype=torch.float64, device=dev)
        k = min(4, m)
        t[:, :k] = torch.where(torch.isfinite(y[:, :k]) & (y[:, :k].abs() < 1e3), y[:, :k], t[:, :k])
        edges = edge_k[ids[q].clamp_min(0)]
        t[..., 1] = torch.where(edges, torch.full_like(t[..., 1], 0.5), t[..., 1])
        out[q] = torch.where((torch.arange(m, device=dev)[None] < n[:, None])[..., None], t, torch.zeros_like(t))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "backward":
        return _exact_backward(prepare(case, seed))
    if kind == "validity":
        return _exact_validity(prepare(case, seed))
    if kind == "infer":
        return _exact_infer(case, seed, prepare(case, seed))
    return None
