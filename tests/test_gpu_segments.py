"""Short segments on the device-wide path (an autotuned plan tries that): one bin and no map each, beside
segments that have one; more of them than 32-bit positions of map cells held."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    from paper_2311_03096_gb300 import ws

    c = ws.Context.get()
    yield c
    c.set_small_max(-1)


def same(ctx, w, offsets, lams, dt):
    from paper_2311_03096_gb300 import ws

    prec = "fp64" if dt == torch.float64 else "fp32comp"
    want = ws.Plan(offsets, dt).forward(w, lams, prec)
    ctx.check(what="one CTA")
    ctx.set_small_max(0)
    plan = ws.Plan(offsets, dt)
    for _ in range(2):
        got = plan.forward(w, lams, prec)
        ctx.check(what="device-wide")
        # the same exact partition; the values round apart
        assert torch.equal(got[1], want[1]) and torch.equal(got[2], want[2])
        tol = 1e-12 if dt == torch.float64 else 1e-5
        assert float((got[0] - want[0]).abs().max()) <= tol * (float(w.abs().max()) + float(lams.max()))


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_short_segments(ctx, dt):
    rng = np.random.default_rng(20)
    lens = np.concatenate([rng.integers(1, 4097, 900), [4096, 4097, 2, 3, 70001, 31, 1400001, 5, 12289, 4096], rng.integers(1, 40, 300)])
    rng.shuffle(lens[:905])
    offsets = np.concatenate([[0], np.cumsum(lens)])
    x = rng.standard_normal(int(offsets[-1]))
    x[rng.random(x.shape[0]) < 0.05] = 0.0
    w = torch.from_numpy(x).cuda().to(dt)
    lams = torch.from_numpy(np.exp(rng.uniform(-7, 1, len(lens)))).cuda()
    same(ctx, w, offsets, lams, dt)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [1, 2, 150, 700, 1350])   # one to nine segments of one tile per CTA
def test_few_segments(ctx, n, dt):
    rng = np.random.default_rng(n)
    lens = rng.integers(1, 4097, n)
    lens[: n // 5] = rng.integers(2049, 6145, n // 5)
    lens[n // 2] = [1, 2049, 4097, 6144, 30000][n % 5]
    offsets = np.concatenate([[0], np.cumsum(lens)])
    w = torch.from_numpy(rng.standard_normal(int(offsets[-1]))).cuda().to(dt)
    lams = torch.from_numpy(np.exp(rng.uniform(-7, 1, n))).cuda()
    same(ctx, w, offsets, lams, dt)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_not_finite(ctx, bad):
    from paper_2311_03096_gb300 import ws

    ctx.set_small_max(0)
    w = torch.ones(5000, device="cuda")
    w[4321] = bad
    ws.Plan([0, 10, 4000, 4500, 5000]).forward(w, torch.ones(4, dtype=torch.float64, device="cuda"))
    assert ctx.status() == ws.WS_ERR_NONFINITE


def test_many_segments(ctx):
    n = 700001
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 90e9:
        pytest.skip("needs 90 GB")
    g = torch.Generator(device="cuda").manual_seed(21)
    w = torch.randn(3 * n, generator=g, device="cuda")
    lams = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    same(ctx, w, 3 * np.arange(n + 1, dtype=np.int64), lams, torch.float32)
