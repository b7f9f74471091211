"""Bins above one CTA's capacity: ties of every size around the capacity and the tile, with no, one and
many neighbours; more heavy values than a bin has splitters; spikes of different values that take the
radix passes; through the sort and through the forward at lambda 0."""
import numpy as np
import pytest

from test_gpu_sort import check as check_sort
from test_gpu_sort import ctx, ws  # noqa: F401  (fixtures)
from test_gpu_way_back import check_lambda_zero

pytestmark = pytest.mark.gpu
DT = [np.float32, np.float64]


def check(ws, ctx, w):  # noqa: F811
    check_sort(ws, ctx, w)
    check_lambda_zero(ws, w)


@pytest.mark.parametrize("dt", DT)
@pytest.mark.parametrize("around", ["nothing", "one each side", "both sides", "below", "both zeros"])
@pytest.mark.parametrize("n", [4095, 4096, 4097, 6144, 6145, 12289, 100003])
def test_one_tie(ws, ctx, n, around, dt):  # noqa: F811
    rng = np.random.default_rng(n)
    v = dt(0.0 if around == "both zeros" else 0.25)
    x = np.full(n, v, dt)
    if around == "one each side":
        x = np.concatenate([x, [np.nextafter(v, dt(-1)), np.nextafter(v, dt(1))]])
    elif around == "both sides":
        x = np.concatenate([x, v + 1e-3 * rng.standard_normal(3000)])
    elif around == "below":
        x = np.concatenate([x, v - 1e-3 * rng.random(5001)])
    elif around == "both zeros":
        x[rng.random(n) < 0.3] = -0.0
        x = np.concatenate([x, 1e-4 * rng.standard_normal(2000)])
    x = x.astype(dt)
    rng.shuffle(x)
    check(ws, ctx, x)


@pytest.mark.parametrize("dt", DT)
@pytest.mark.parametrize("copies", [300, 4200, 7000])
@pytest.mark.parametrize("span", [1e-5, 1.0])
def test_many_heavy_values(ws, ctx, copies, span, dt):  # noqa: F811
    """70 values, in one bin or spread, each with `copies` copies, and other weights between them."""
    rng = np.random.default_rng(copies)
    v = 1.0 + span * np.sort(rng.random(70))
    x = np.concatenate([np.repeat(v, copies), 1.0 + span * rng.random(20000), rng.standard_normal(50000)]).astype(dt)
    rng.shuffle(x)
    check(ws, ctx, x)


@pytest.mark.parametrize("spikes", [1, 3])
def test_spikes_of_different_values(ws, ctx, spikes):  # noqa: F811
    """More different values than the splitters cut into classes of one CTA."""
    rng = np.random.default_rng(9)
    d = 1300000
    x = rng.integers(0, spikes, d) + 1.0 + rng.integers(0, 10 ** 6, d) * 2.0 ** -50
    x[:5] = [-1e30, 1e30, 0.0, 0.5, 1.0]
    rng.shuffle(x)
    check_sort(ws, ctx, x)


@pytest.mark.parametrize("dt", DT)
def test_segments_with_and_without(ws, ctx, dt):  # noqa: F811
    """Oversize bins of several segments in one call, beside segments that have none."""
    import torch

    rng = np.random.default_rng(10)
    lens = [5000, 4097, 70001, 9000, 1500000, 4098]
    parts = [rng.standard_normal(n).astype(dt) for n in lens]
    for i, share in ((1, 1.0), (2, 0.4), (4, 0.01), (5, 0.999)):
        parts[i][rng.random(lens[i]) < share] = dt(0.5 * i)
    w = np.concatenate(parts)
    plan = ws.Plan(np.concatenate([[0], np.cumsum(lens)]), torch.from_numpy(w).dtype)
    lam = torch.zeros(len(lens), dtype=torch.float64, device="cuda")
    x = torch.from_numpy(w).cuda()
    for _ in range(2):
        out, ids, nc = plan.forward(x, lam, "fp64" if dt == np.float64 else "fp32comp")
        ctx.check(what="forward")
        got = np.split(ids.cpu().numpy(), np.cumsum(lens)[:-1])
        for g, p, n in zip(got, parts, nc.cpu().numpy()):
            u, inv = np.unique(p, return_inverse=True)
            assert np.array_equal(g, inv) and n == len(u)


@pytest.mark.parametrize("d", [70001, 1500001])
def test_captured_call_with_and_without_ties(ws, ctx, d):  # noqa: F811
    """One captured call replayed on values with heavy ties, without, and with other ones."""
    import torch

    g = torch.Generator(device="cuda").manual_seed(14)
    base = torch.randn(d, generator=g, device="cuda")
    r = torch.rand(d, generator=g, device="cuda")
    inputs = [torch.where(r < p, torch.full_like(base, v), base) for p, v in ((0.5, 0.0), (0.0, 0.0), (0.9, 1.5), (0.3, -0.25))]
    w = base.clone()
    out, ids = torch.empty_like(w), torch.empty(d, dtype=torch.int32, device="cuda")
    nc = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws.prox(w, 0.01, out=out, id_out=ids, n_clusters=nc)   # (the plan is made outside the capture)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ws.prox(w, 0.01, out=out, id_out=ids, n_clusters=nc)
    for x in inputs + inputs[::-1]:
        w.copy_(x)
        graph.replay()
        torch.cuda.synchronize()
        ctx.check(what="replay")
        want = ws.prox(x, 0.01)
        assert torch.equal(out, want[0]) and torch.equal(ids, want[1]) and torch.equal(nc, want[2])
