"""What is timed when the speed of the framework is measured: the proximal map
and its backward, R(w) and the proximal training step, each through the entry
points that a program calls (paper_2311_03096_gb300.ws and .train).

Sizes are those of the repository's workloads (inputs.py, bench.py, the tests):
FP64 vectors of 4096 weights, FP32 vectors up to 2^26 weights with 10 % exact
duplicates, the rows and layers of the MLP 3072-4096-4096-10 with
Kaiming-uniform weights, and batches of segments with log-uniform lengths in
[16, 2^20].  lambda is 1e-2, 1 or 1e2 for N(0, 1) vectors and
LogUniform[1e-3, 1] per segment in batches.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_03096_gb300 import inputs, train, ws

MLP = inputs.MLP_SIZES
VEC_MAX = 2 ** 26
DTYPES = {"f32": torch.float32, "f64": torch.float64}


def listed():
    return [
        # a small FP64 vector (one neuron's weights in a study that wants FP64): latency
        {"name": "vec_f64_4096", "kind": "vec", "d": 4096, "dtype": "f64", "prec": "fp64", "lam": 0.1,
         "values": "normal"},
        # the output layer of the MLP as one vector, weight sharing + l1 with rewinding: a
        # small device-wide call, where launches count
        {"name": "l1_f32_40960", "kind": "l1", "d": 40960, "dtype": "f32", "prec": "fp32comp", "lam": 1e-2,
         "beta": 1e-3, "rho": 0.5, "values": "kaiming"},
        # a layer of odd size as one vector
        {"name": "vec_f32_1000003", "kind": "vec", "d": 1000003, "dtype": "f32", "prec": "fp32comp", "lam": 1e-2,
         "values": "duplicates"},
        # a whole hidden layer's worth of weights as one vector, medium lambda
        {"name": "vec_f32_2e24", "kind": "vec", "d": 2 ** 24, "dtype": "f32", "prec": "fp32comp", "lam": 1.0,
         "values": "duplicates"},
        # the largest single vector of the benchmark, short clusters
        {"name": "vec_f32_2e26", "kind": "vec", "d": 2 ** 26, "dtype": "f32", "prec": "fp32comp", "lam": 1e-2,
         "values": "duplicates"},
        # FP64 storage and arithmetic on a large vector of odd size
        {"name": "vec_f64_4194001", "kind": "vec", "d": 4194001, "dtype": "f64", "prec": "fp64", "lam": 1.0,
         "values": "duplicates"},
        # every output-neuron row of the MLP, one lambda per row (a planned batch)
        {"name": "rows_mlp", "kind": "rows", "seed_lam": 7},
        # thousands of uneven segments: layers of many sizes in one planned call
        {"name": "uneven_1024", "kind": "uneven", "n_seg": 1024, "lo": 16, "hi": 2 ** 20},
        # backward of a large vector, with the derivative with respect to lambda
        {"name": "bwd_f32_2e24", "kind": "bwd", "d": 2 ** 24, "dtype": "f32", "lam": 1e-2, "values": "duplicates"},
        # differentiable prox of a weight matrix, per row: forward and backward through autograd
        {"name": "autograd_4096x3072", "kind": "autograd", "rows": 4096, "cols": 3072, "lam": 1e-2},
        # the penalty and the weight-sharing measure of a layer whose weights are already shared
        {"name": "R_shared_4096x3072", "kind": "R", "d": 4096 * 3072, "dtype": "f32", "lam": 1.0},
        # one proximal SGD step of the MLP (batch 256): what a training loop pays
        {"name": "train_step", "kind": "train", "batch": 256, "alpha": 1e-3},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["vec", "vec", "vec", "vec64", "vec64", "l1", "rows", "uneven", "bwd", "autograd", "R", "train"])
    values = rng.choice(["duplicates", "normal", "kaiming"])
    lam = _log_uniform(rng, 1e-2, 1e2) if values != "kaiming" else _log_uniform(rng, 1e-3, 1e-1)
    if kind == "vec":
        return {"kind": "vec", "d": int(_log_uniform(rng, 1000, VEC_MAX)), "dtype": "f32",
                "prec": rng.choice(["fp32comp", "fp32comp", "fp64"]), "lam": lam, "values": values}
    if kind == "vec64":
        return {"kind": "vec", "d": int(_log_uniform(rng, 1000, 2 ** 23)), "dtype": "f64", "prec": "fp64",
                "lam": lam, "values": values}
    if kind == "l1":
        return {"kind": "l1", "d": int(_log_uniform(rng, 4097, 2 ** 24)), "dtype": "f32", "prec": "fp32comp",
                "lam": lam, "beta": _log_uniform(rng, 1e-4, 1e-1), "rho": rng.choice([0.0, 0.5, 1.0]),
                "values": values}
    if kind == "rows":
        return {"kind": "rows", "seed_lam": rng.randrange(1 << 20), "rows": int(_log_uniform(rng, 10, 8192)),
                "cols": rng.randrange(64, 4097)}
    if kind == "uneven":
        return {"kind": "uneven", "n_seg": int(_log_uniform(rng, 16, 1024)), "lo": 16, "hi": 2 ** 20}
    if kind == "bwd":
        return {"kind": "bwd", "d": int(_log_uniform(rng, 1000, 2 ** 25)), "dtype": rng.choice(["f32", "f32", "f64"]),
                "lam": lam, "values": values}
    if kind == "autograd":
        return {"kind": "autograd", "rows": int(_log_uniform(rng, 10, 4096)), "cols": rng.randrange(64, 4097),
                "lam": _log_uniform(rng, 1e-3, 1.0)}
    if kind == "R":
        return {"kind": "R", "d": int(_log_uniform(rng, 1000, 2 ** 25)), "dtype": "f32", "lam": lam}
    return {"kind": "train", "batch": rng.randrange(32, 257), "alpha": _log_uniform(rng, 1e-4, 1e-2)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _vector(case, seed):
    """The weights of a single vector; "duplicates": 10 % of the positions are
    exact copies of others; "kaiming": uniform in +-sqrt(6 / 4096)."""
    d, dt = case["d"], DTYPES[case["dtype"]]
    g = _gen(seed)
    values = case.get("values", "normal")
    if values == "kaiming":
        b = math.sqrt(6.0 / 4096)
        return torch.rand(d, generator=g, device="cuda", dtype=dt).mul_(2 * b).sub_(b)
    w = torch.randn(d, generator=g, device="cuda", dtype=dt)
    if values == "duplicates":
        m = max(d // 10, 1)
        dst = torch.randint(0, d - m + 1, (1,), generator=g, device="cuda")
        src = torch.randint(0, d, (m,), generator=g, device="cuda")
        pos = (torch.arange(m, device="cuda") * 9 + dst) % d   # (9 m < d: distinct positions)
        w[pos] = w[src]
    return w


def _log_uniform_lams(n, seed):
    g = _gen(seed)
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    return torch.exp(u * math.log(1e3) + math.log(1e-3))


def _layout(case, seed):
    """(offsets, values, lambdas) of a batched case.  The layout is the program's
    own (the model's shapes): it does not depend on the seed."""
    g = _gen(seed)
    if case["kind"] == "rows":
        if "rows" in case:
            shapes = [(case["rows"], case["cols"])]
        else:
            shapes = [(o, i) for i, o in zip(MLP[:-1], MLP[1:])]
        lens = np.concatenate([np.full(r, c, np.int64) for r, c in shapes])
        parts = []
        for r, c in shapes:
            b = math.sqrt(6.0 / c)
            parts.append(torch.rand(r * c, generator=g, device="cuda").mul_(2 * b).sub_(b))
        values = torch.cat(parts)
        lams = _log_uniform_lams(lens.shape[0], case["seed_lam"] + seed)
    else:
        lens = inputs.log_uniform_lengths(case["n_seg"], case["lo"], case["hi"], 101)
        values = torch.randn(int(lens.sum()), generator=g, device="cuda")
        lams = _log_uniform_lams(lens.shape[0], seed + 303)
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return offsets, values, lams


def _matrix(case, seed):
    b = math.sqrt(6.0 / case["cols"])
    g = _gen(seed)
    w = torch.rand(case["rows"], case["cols"], generator=g, device="cuda").mul_(2 * b).sub_(b)
    gy = torch.randn(case["rows"], case["cols"], generator=g, device="cuda")
    return w, gy


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("vec", "l1"):
        return {"case": case, "w": _vector(case, seed)}
    if kind in ("rows", "uneven"):
        offsets, values, lams = _layout(case, seed)
        return {"case": case, "plan": ws.Plan(offsets, torch.float32), "values": values, "lams": lams}
    if kind == "bwd":
        w = _vector(case, seed)
        prec = "fp64" if case["dtype"] == "f64" else "fp32comp"
        _, ids, _ = ws.prox(w, case["lam"], prec)
        return {"case": case, "g": torch.randn(case["d"], generator=_gen(seed + 1), device="cuda", dtype=w.dtype),
                "ids": ids}
    if kind == "autograd":
        w, gy = _matrix(case, seed)
        return {"case": case, "w": w.requires_grad_(True), "gy": gy}
    if kind == "R":
        w = _vector({**case, "values": "normal"}, seed)
        out, _, _ = ws.prox(w, case["lam"])
        return {"case": case, "w": out}
    x, y = inputs.images(case["batch"], seed)
    return {"case": case, "mlp": train.ProxMLP(seed=seed, alpha=case["alpha"]),
            "x": torch.from_numpy(x).cuda(), "y": torch.from_numpy(y).cuda()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "vec":
        return ws.prox(state["w"], case["lam"], case["prec"])
    if kind == "l1":
        return ws.prox_l1(state["w"], case["lam"], case["beta"], case["rho"], prec=case["prec"])
    if kind in ("rows", "uneven"):
        return state["plan"].forward(state["values"], state["lams"])
    if kind == "bwd":
        return ws.prox_backward(state["g"], state["ids"]), ws.prox_dlambda(state["g"], state["ids"])
    if kind == "autograd":
        w = state["w"]
        y = ws.WSProx.apply(w, case["lam"])
        (gw,) = torch.autograd.grad(y, w, state["gy"])
        return y.detach(), gw
    if kind == "R":
        return ws.R(state["w"])
    mlp = state["mlp"]
    loss = mlp.step(state["x"], state["y"])
    return loss, mlp.flat, mlp.ids, mlp.n_clusters


def work(case):
    """Bytes: inputs read once and outputs written once; flops: one shift and one
    sum per weight (the path is a sort and a merge, not arithmetic)."""
    kind = case["kind"]
    if kind in ("vec", "l1"):
        s = 8 if case["dtype"] == "f64" else 4
        return {"bytes": case["d"] * (2 * s + 4), "flops": 2 * case["d"]}
    if kind == "rows":
        n = case["rows"] * case["cols"] if "rows" in case else sum(a * b for a, b in zip(MLP[:-1], MLP[1:]))
        return {"bytes": 12 * n, "flops": 2 * n}
    if kind == "uneven":
        n = int(inputs.log_uniform_lengths(case["n_seg"], case["lo"], case["hi"], 101).sum())
        return {"bytes": 12 * n, "flops": 2 * n}
    if kind == "bwd":
        s = 8 if case["dtype"] == "f64" else 4
        return {"bytes": case["d"] * (2 * s + 4), "flops": 2 * case["d"]}
    if kind == "autograd":
        n = case["rows"] * case["cols"]
        return {"bytes": 16 * n, "flops": 4 * n}
    if kind == "R":
        return {"bytes": 4 * case["d"], "flops": 2 * case["d"]}
    n = sum(a * b for a, b in zip(MLP[:-1], MLP[1:]))
    # forward and weight-gradient products of every layer, the input gradient of all but the first
    macs = 3 * n - MLP[0] * MLP[1]
    # weights read, updated weights and ids written, the batch read
    return {"bytes": 12 * n + 4 * case["batch"] * MLP[0], "flops": 2 * case["batch"] * macs + 2 * n}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _pool(w, lens, lams, group=None):
    """Isotonic regression of the shifted sorted weights of every segment, in 64
    bits, by rounds that merge every run of adjacent violators.  Returns, for
    every weight in its own order: mean weight and mean shift of its cluster, and
    its cluster's number (over the whole batch)."""
    n = w.shape[0]
    dev = w.device
    lens_t = torch.as_tensor(lens, device=dev, dtype=torch.int64)
    x, order = torch.sort(w.double())
    if lens_t.shape[0] == 1:
        d = n
        shift = lams[0] * (d - 1 - 2 * torch.arange(n, device=dev, dtype=torch.float64)) / max(d - 1, 1)
        first = None
    else:
        seg = torch.repeat_interleave(torch.arange(lens_t.shape[0], device=dev, dtype=torch.int32), lens_t)
        s2, o2 = torch.sort(seg[order], stable=True)
        x, order = x[o2], order[o2]
        del o2
        starts = torch.cumsum(lens_t, 0) - lens_t
        sl = s2.long()
        d = lens_t[sl].double()
        j = torch.arange(n, device=dev, dtype=torch.float64) - starts[sl].double()
        shift = lams[sl] * (d - 1 - 2 * j) / torch.clamp(d - 1, min=1)
        first = s2
        del sl, d, j
    cx, cv = x, shift
    cnt = torch.ones(n, device=dev, dtype=torch.float64)
    label = torch.arange(n, device=dev)   # block of every sorted position
    seg_of = first
    while True:
        m = (cx + cv) / cnt
        hit = m[:-1] >= m[1:]
        if seg_of is not None:
            hit &= seg_of[:-1] == seg_of[1:]
        if not bool(hit.any()):
            break
        new = torch.zeros(m.shape[0], device=dev, dtype=torch.int64)
        new[1:] = torch.cumsum(~hit, 0)
        k = int(new[-1]) + 1
        cx = torch.zeros(k, device=dev, dtype=torch.float64).index_add_(0, new, cx)
        cv = torch.zeros(k, device=dev, dtype=torch.float64).index_add_(0, new, cv)
        cnt = torch.zeros(k, device=dev, dtype=torch.float64).index_add_(0, new, cnt)
        if seg_of is not None:
            seg_of = torch.zeros(k, device=dev, dtype=seg_of.dtype).index_copy_(0, new, seg_of)
        label = new[label]
    back = torch.empty_like(label)
    back[order] = label
    return (cx / cnt)[back], (cv / cnt)[back], back


def _cluster_mean(g, cid):
    k = int(cid.max()) + 1
    s = torch.zeros(k, device=g.device, dtype=torch.float64).index_add_(0, cid, g.double())
    c = torch.zeros(k, device=g.device, dtype=torch.float64).index_add_(0, cid, torch.ones_like(g, dtype=torch.float64))
    return (s / c)[cid]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("vec", "l1", "bwd"):
        w = _vector(case, seed)
        lam = torch.tensor([case["lam"]], dtype=torch.float64, device="cuda")
        x, v, cid = _pool(w, [case["d"]], lam)
        if kind == "vec":
            return [x + v, None, None]
        if kind == "l1":
            s = x + v
            y = x + (1.0 - case["rho"]) * (v - case["beta"] * torch.sign(s))
            return [torch.where(s.abs() < case["beta"], torch.zeros_like(s), y), None, None]
        g = torch.randn(case["d"], generator=_gen(seed + 1), device="cuda", dtype=w.dtype)
        d = case["d"]
        # d out / d lambda: the mean of (d - 1 - 2 j)/(d - 1) over the cluster's sorted positions
        vel = v / case["lam"]
        return [_cluster_mean(g, cid), (g.double() * vel).sum().reshape(1) if d > 1 else None]
    if kind in ("rows", "uneven"):
        offsets, values, lams = _layout(case, seed)
        x, v, _ = _pool(values, np.diff(offsets), lams)
        return [x + v, None, None]
    if kind == "autograd":
        w, gy = _matrix(case, seed)
        lams = torch.full((case["rows"],), case["lam"], dtype=torch.float64, device="cuda")
        x, v, cid = _pool(w.reshape(-1), np.full(case["rows"], case["cols"]), lams)
        return [(x + v).reshape(w.shape), _cluster_mean(gy.reshape(-1), cid).reshape(w.shape)]
    return None   # R: of weights that the framework's own prox has shared; train: a whole model's step
