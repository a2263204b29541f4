"""The work this library is measured on: one pass of each public entry point
over the range of sizes, cost structures and options its users run.

Dense solves from the smallest instance to the largest configuration, the
packed batch, the learned warm start and the predictor's training step,
sparse graphs, grid max-flow and the dual certificate. Inputs are drawn from
the seed on the GPU (search-window graphs on the host, by ``synth``).

The optimal cost of an instance is unique, its optimal matching need not be:
among equal costs the lock-free bids of two runs may settle on different
optima. Where costs are so fine that two optimal matchings are out of the
question (independent costs over at least ``16384 n`` values), a solve returns its
matching beside the cost. The duals of ``dual_certificate`` and the source
side of ``maxflow_grid`` do not depend on which optimum was found.
"""

import ctypes
import math

import numpy as np
import torch

import paper_1110_6231_gb300 as la
from paper_1110_6231_gb300 import learn, synth

DEV = "cuda"


def listed():
    return [
        # a frame-to-frame tracker's association step: the smallest call, latency is everything
        {"name": "solve-uniform-n64", "kind": "uniform", "n": 64, "hi": (1 << 20) - 1},
        # the configured small instance: 8-bit-like scores, 16-bit costs on one CTA
        {"name": "solve-uniform-n256-c1000", "kind": "uniform", "n": 256, "hi": 1000},
        # optical flow on a thousand features, every option at its default
        {"name": "solve-geometric-n1024", "kind": "geometric", "n": 1024},
        # independent costs at the configured size, with the options the README gives for it
        {"name": "solve-uniform-n4096-c2^20", "kind": "uniform", "n": 4096, "hi": (1 << 20) - 1, "alpha": 48,
         "alpha_fine": 4},
        # the headline: the largest single matrix (256 MiB), with the README's options for it
        {"name": "solve-geometric-n8192", "kind": "geometric", "n": 8192, "price_updates": 4, "tail_threshold": 128},
        # a packed batch of uneven instances, half uniform and half geometric (training data, many frames)
        {"name": "batch-2000-n16-1024", "kind": "batch", "count": 2000, "lo": 16, "hi_n": 1024},
        # a solve warm-started by the predictor, at the size it was trained for
        {"name": "warm-geometric-n1024", "kind": "warm", "n": 1024},
        # one training step of the predictor on 64 instances (learn.train's batch)
        {"name": "train-step-64", "kind": "train", "count": 64, "lo": 256, "hi_n": 1024},
        # sparse graphs: random arcs at the configured size; the search-window graph of optical flow
        {"name": "sparse-uniform-n65536-d32", "kind": "sparse-uniform", "n": 65536, "degree": 32},
        {"name": "sparse-geometric-n16384", "kind": "sparse-geometric", "n": 16384},
        # graph-cut segmentation of a megapixel image
        {"name": "gridcut-1024x1024", "kind": "cut", "H": 1024, "W": 1024},
        # the proof that comes with an optimum (and the predictor's training targets)
        {"name": "certificate-geometric-n2048", "kind": "certificate", "n": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["uniform", "uniform", "geometric", "geometric", "batch", "warm", "train", "sparse-uniform",
                       "sparse-geometric", "cut", "cross", "certificate"])
    if kind == "uniform":
        n = _log_int(rng, 32, 4096)
        c = {"kind": kind, "n": n, "hi": rng.choice([1000, 65535, (1 << 20) - 1, (1 << 28) - 1 if n < 2048 else (1 << 26) - 1])}
        if n >= 2048:
            c.update(alpha=48, alpha_fine=4)
        return c
    if kind == "geometric":
        n = _log_int(rng, 128, 8192)
        c = {"kind": kind, "n": n}
        if n >= 4096:
            c.update(price_updates=4, tail_threshold=128)
        return c
    if kind == "batch":
        return {"kind": kind, "count": _log_int(rng, 64, 2000), "lo": rng.randint(8, 64), "hi_n": _log_int(rng, 128, 1024)}
    if kind == "warm":
        return {"kind": kind, "n": _log_int(rng, 256, 4096)}
    if kind == "train":
        return {"kind": kind, "count": _log_int(rng, 8, 64), "lo": 256, "hi_n": rng.randint(512, 1024)}
    if kind == "sparse-uniform":
        return {"kind": kind, "n": _log_int(rng, 2048, 65536), "degree": rng.randint(8, 32)}
    if kind == "sparse-geometric":
        return {"kind": kind, "n": _log_int(rng, 2048, 16384)}
    if kind in ("cut", "cross"):
        top = 1024 if kind == "cut" else 512
        return {"kind": kind, "H": _log_int(rng, 96, top), "W": _log_int(rng, 96, top)}
    return {"kind": "certificate", "n": _log_int(rng, 128, 4096)}


# ------------------------------------------------------------------ inputs


def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + 7919 * stream) & 0x7FFFFFFFFFFF)
    return g


def _uniform(n, hi, g):
    return torch.randint(0, hi + 1, (n, n), generator=g, device=DEV, dtype=torch.int32)


def _geometric(n, g, sigma=0.01, scale=1.0e4):
    """rint(scale |a_i - b_j|^2) with b the points a permuted and jittered (synth.geometric_costs' recipe)."""
    a = torch.rand((n, 2), generator=g, device=DEV, dtype=torch.float64)
    p = torch.randperm(n, generator=g, device=DEV)
    b = a[p] + sigma * torch.randn((n, 2), generator=g, device=DEV, dtype=torch.float64)
    out = torch.empty((n, n), dtype=torch.int32, device=DEV)
    for r in range(0, n, 1024):
        d = a[r:r + 1024, None, :] - b[None, :, :]
        out[r:r + 1024] = torch.round((d * d).sum(-1) * scale).to(torch.int32)
    return out


def _grid_cut(H, W, g, disks=12, noise=0.12, data=1000.0, smooth=300.0, sigma_edge=0.1):
    """Bright disks on a dark noisy image, segmented (synth.grid_cut's recipe)."""
    side = float(min(H, W))
    d = torch.rand((disks, 3), generator=g, device=DEV, dtype=torch.float64)
    ii = torch.arange(H, device=DEV, dtype=torch.float64)[:, None] + 0.5
    jj = torch.arange(W, device=DEV, dtype=torch.float64)[None, :] + 0.5
    inside = torch.zeros((H, W), dtype=torch.bool, device=DEV)
    for k in range(disks):
        r = (0.03 + 0.12 * d[k, 2]) * side
        inside |= (ii - d[k, 0] * H) ** 2 + (jj - d[k, 1] * W) ** 2 <= r * r
    img = torch.where(inside, 0.8, 0.2) + noise * torch.randn((H, W), generator=g, device=DEV, dtype=torch.float64)
    src = torch.round(data * (img - 0.2) ** 2).to(torch.int32)
    snk = torch.round(data * (img - 0.8) ** 2).to(torch.int32)
    cap = torch.zeros((4, H, W), dtype=torch.int32, device=DEV)
    inv = -1.0 / (2.0 * sigma_edge * sigma_edge)
    w = torch.round(smooth * torch.exp(inv * (img[:, 1:] - img[:, :-1]) ** 2)).to(torch.int32)
    cap[0, :, :-1], cap[1, :, 1:] = w, w
    w = torch.round(smooth * torch.exp(inv * (img[1:] - img[:-1]) ** 2)).to(torch.int32)
    cap[2, :-1], cap[3, 1:] = w, w
    return cap, src, snk


def _grid_crossing(H, W, g, hi=100):
    """Flow from the left column to the right one (synth.grid_crossing's recipe)."""
    cap = torch.randint(1, hi + 1, (4, H, W), generator=g, device=DEV, dtype=torch.int32)
    cap[0, :, -1] = 0
    cap[1, :, 0] = 0
    cap[2, -1] = 0
    cap[3, 0] = 0
    src = torch.zeros((H, W), dtype=torch.int32, device=DEV)
    snk = torch.zeros_like(src)
    src[:, 0] = 100 * hi
    snk[:, -1] = 100 * hi
    return cap, src, snk


def _sparse_uniform(n, degree, g, hi=10_000):
    """Arcs to `degree` random columns and to a planted partner, duplicates merged (synth.sparse_uniform's recipe)."""
    rows = torch.arange(n, device=DEV)
    key = torch.cat([rows * n + torch.randperm(n, generator=g, device=DEV),
                     rows.repeat_interleave(degree) * n
                     + torch.randint(0, n, (n * degree,), generator=g, device=DEV)]).unique()
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    costs = torch.randint(0, hi + 1, key.shape, generator=g, device=DEV, dtype=torch.int32)
    return [row_ptr.int(), (key % n).int(), costs]


def _sizes(case, seed):
    r = np.random.default_rng(seed)
    lo, hi = math.log(case["lo"]), math.log(case["hi_n"])
    return np.clip(np.floor(np.exp(r.uniform(lo, hi, case["count"]))), case["lo"], case["hi_n"]).astype(np.int64)


def _train_inputs(case, seed):
    """A batch as learn.train gathers it, in the middle of training: features with the distributions la_features
    gives, targets that depend on them, weights, and Adam's moments."""
    r = np.random.default_rng(seed)
    sizes = r.integers(case["lo"], case["hi_n"] + 1, size=case["count"])
    N = int(sizes.sum())
    seg = np.zeros(len(sizes) + 1, dtype=np.int32)
    seg[1:] = np.cumsum(sizes)
    g = _gen(seed, 1)
    f = torch.zeros((N, la.LA_PRED_FEATURES_PADDED), dtype=torch.float32, device=DEV)
    z = torch.randn((N, 4), generator=g, device=DEV)
    f[:, 0] = z[:, 0]
    f[:, 1] = z[:, 1].abs()
    f[:, 2] = 0.5 * z[:, 0] + 0.5 * z[:, 2]
    f[:, 3] = z[:, 2].abs()
    f[:, 4] = torch.log1p(torch.randint(0, 5, (N,), generator=g, device=DEV).float())
    f[:, 5] = z[:, 3]
    ln = torch.from_numpy(np.repeat(np.log(sizes) * 0.1, sizes).astype(np.float32)).to(DEV)
    f[:, 6] = 0.1
    f[:, 7] = ln
    t = (-0.8 * f[:, 0] + 0.4 * f[:, 1] - 0.3 * f[:, 2]
         + 0.2 * torch.randn((N,), generator=g, device=DEV)).contiguous()
    P = torch.from_numpy(learn.init_params(seed)).to(DEV)
    m = 1e-3 * torch.randn(P.shape, generator=g, device=DEV)
    v = (0.02 * (1.0 + torch.rand(P.shape, generator=g, device=DEV))) ** 2
    return {"P": P, "m": m, "v": v, "f": f, "t": t, "seg": torch.from_numpy(seg).to(DEV), "I": len(sizes), "N": N,
            "step": 200, "lr": 2e-3}


_SOLVE_OPTIONS = ("alpha", "alpha_fine", "price_updates", "tail_threshold")


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k}
    if k in ("uniform", "geometric"):
        n = case["n"]
        s["C"] = _uniform(n, case["hi"], _gen(seed, 0)) if k == "uniform" else _geometric(n, _gen(seed, 0))
        s["options"] = {o: case[o] for o in _SOLVE_OPTIONS if o in case}
        s["unique"] = k == "uniform" and case["hi"] + 1 >= 16384 * n
    elif k == "batch":
        ns = _sizes(case, seed)
        off = np.zeros(len(ns), dtype=np.int64)
        off[1:] = np.cumsum(ns ** 2)[:-1]
        g = _gen(seed, 0)
        flat = torch.randint(0, 10_001, (int((ns ** 2).sum()),), generator=g, device=DEV, dtype=torch.int32)
        for i in range(1, len(ns), 2):
            n = int(ns[i])
            flat[int(off[i]):int(off[i]) + n * n] = _geometric(n, g).view(-1)
        s.update(costs=flat, offsets=torch.from_numpy(off).to(DEV), ns=torch.from_numpy(ns.astype(np.int32)).to(DEV),
                 options=la.batch_options(max_n=case["hi_n"]))
    elif k == "warm":
        s["C"] = _geometric(case["n"], _gen(seed, 0))
        s["W"] = torch.from_numpy(np.fromfile(learn.DEFAULT_WEIGHTS, dtype=np.float32)).to(DEV)
    elif k == "train":
        s.update(_train_inputs(case, seed))
        s["grad"] = torch.empty_like(s["P"])
        s["loss"] = ctypes.c_float(0.0)
    elif k in ("sparse-uniform", "sparse-geometric"):
        s["csr"] = (_sparse_uniform(case["n"], case["degree"], _gen(seed, 0)) if k == "sparse-uniform"
                    else [torch.from_numpy(x).to(DEV) for x in synth.sparse_geometric(case["n"], seed)])
    elif k in ("cut", "cross"):
        make = _grid_cut if k == "cut" else _grid_crossing
        s["grid"] = make(case["H"], case["W"], _gen(seed, 0))
    else:
        s["C"] = _geometric(case["n"], _gen(seed, 0))
        s["match"] = la.solve(s["C"]).match
    return s


def run(state):
    k = state["kind"]
    if k in ("uniform", "geometric"):
        sol = la.solve(state["C"], **state["options"])
        return {"cost": sol.cost, "match": sol.match} if state["unique"] else {"cost": sol.cost}
    if k == "batch":
        sol = la.solve_batched(state["costs"], state["offsets"], state["ns"], options=state["options"])
        return {"costs": sol.costs, "status": sol.status}
    if k == "warm":
        return {"cost": la.solve_warm(state["C"], state["W"]).cost}
    if k == "train":
        s = state
        rc = la.la_predictor_train_step(s["P"], s["m"], s["v"], s["f"], s["t"], s["seg"], s["I"], s["N"], s["step"],
                                        s["lr"], 0.0, None, s["grad"], ctypes.byref(s["loss"]))
        if rc != la.LA_OK:
            raise la.LaError(rc, "la_predictor_train_step")
        return {"loss": float(s["loss"].value), "grad": s["grad"], "params": s["P"], "m": s["m"], "v": s["v"]}
    if k in ("sparse-uniform", "sparse-geometric"):
        return {"cost": la.solve_sparse(*state["csr"]).cost}
    if k in ("cut", "cross"):
        r = la.maxflow_grid(*state["grid"])
        return {"flow": r.flow, "cut": r.cut}
    u, v = la.dual_certificate(state["C"], state["match"])
    return {"u": u, "v": v}


def _mean_log(lo, hi, power):
    """Mean of n^power for n spread over its logarithm on [lo, hi]."""
    return (hi ** power - lo ** power) / (power * math.log(hi / lo))


def work(case):
    """Each input read once and each output written once; the products of the training step."""
    k = case["kind"]
    if k in ("uniform", "geometric", "warm"):
        n = case["n"]
        return {"bytes": 4 * n * n + 4 * n + 8, "flops": 0}
    if k == "batch":
        n2, n1 = _mean_log(case["lo"], case["hi_n"], 2), _mean_log(case["lo"], case["hi_n"], 1)
        return {"bytes": case["count"] * (4 * n2 + 4 * n1 + 24), "flops": 0}
    if k == "train":
        N, H, F = case["count"] * (case["lo"] + case["hi_n"]) / 2, la.LA_PRED_WIDTH, la.LA_PRED_FEATURES
        return {"bytes": N * (4 * la.LA_PRED_FEATURES_PADDED + 4) + 4 * 7 * la.LA_PRED_PARAMS,
                "flops": 2 * N * (2 * F * H + 3 * 2 * H * H + 3 * H)}
    if k == "sparse-uniform":
        n = case["n"]
        return {"bytes": 8 * n * (case["degree"] + 1) + 8 * n, "flops": 0}
    if k == "sparse-geometric":
        n = case["n"]
        return {"bytes": 8 * n * 36 + 8 * n, "flops": 0}
    if k in ("cut", "cross"):
        N = case["H"] * case["W"]
        return {"bytes": 24 * N + N, "flops": 0}
    n = case["n"]
    return {"bytes": 4 * n * n + 4 * n + 16 * n, "flops": 0}


def exact(case, seed):
    """The training step in 64 bits: forward, the variance loss, its gradients and Adam. Everything else is whole numbers."""
    if case["kind"] != "train":
        return None
    s = _train_inputs(case, seed)
    F, H, o = la.LA_PRED_FEATURES_PADDED, la.LA_PRED_WIDTH, la.LA_PRED_HEADER
    P = s["P"].double().requires_grad_(True)
    at = o
    parts = []
    for shape in ((F, H), (H,), (2 * H, H), (H,), (H, 8), (8,)):
        size = math.prod(shape)
        parts.append(P[at:at + size].view(shape))
        at += size
    W1, b1, W2, b2, W3, b3 = parts
    seg = s["seg"].long()
    n = (seg[1:] - seg[:-1]).double()
    which = torch.repeat_interleave(torch.arange(s["I"], device=DEV), seg[1:] - seg[:-1])

    def seg_mean(x):
        return torch.zeros((s["I"],) + x.shape[1:], dtype=x.dtype, device=DEV).index_add(0, which, x) / (
            n.view(-1, *[1] * (x.dim() - 1)))

    h1 = torch.relu(s["f"].double() @ W1 + b1)
    h2 = torch.relu(h1 @ W2[:H] + (seg_mean(h1) @ W2[H:])[which] + b2)
    d = (h2 @ W3 + b3)[:, 0] - s["t"].double()
    d = d - seg_mean(d)[which]
    loss = seg_mean(d * d).mean()
    loss.backward()
    g = P.grad
    m = 0.9 * s["m"].double() + 0.1 * g
    v = 0.999 * s["v"].double() + 0.001 * g * g
    new = P.detach() - s["lr"] * (m / (1 - 0.9 ** s["step"])) / ((v / (1 - 0.999 ** s["step"])).sqrt() + 1e-8)
    keep = torch.arange(P.numel(), device=DEV) < o       # the header is no weight
    return {"loss": float(loss.detach()), "grad": g, "params": torch.where(keep, P.detach(), new),
            "m": torch.where(keep, s["m"].double(), m), "v": torch.where(keep, s["v"].double(), v)}
