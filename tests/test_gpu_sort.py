"""The distribution sort of the device-wide path, bit for bit against numpy:
bins at their edges, one and two partition passes, distributions that the
sampled map resolves well or not at all, and ties beyond one bin's capacity."""
import numpy as np
import pytest
import torch

from paper_2311_03096_gb300 import inputs

pytestmark = pytest.mark.gpu
UINT = {np.float32: np.uint32, np.float64: np.uint64}
TT = {np.float32: torch.float32, np.float64: torch.float64}


@pytest.fixture(scope="module")
def ws():
    from paper_2311_03096_gb300 import ws as m

    return m


@pytest.fixture
def ctx(ws):
    c = ws.Context.get()
    c.set_small_max(0)
    yield c
    c.set_small_max(-1)


def draw(kind, d, dt, seed=5):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(d)
    if kind == "duplicates":
        return inputs.with_duplicates(x.astype(dt), 0.1, seed)
    if kind == "narrow":            # one binade, a sliver of it, and one far outlier
        x = 1.0 + 1e-4 * x
        x[d // 3] = -3e30
    elif kind == "sparse":          # half zeros of both signs (one heavy tie), the rest spread
        x[rng.random(d) < 0.5] = 0.0
        x[rng.random(d) < 0.1] *= -0.0
    elif kind == "few":             # a handful of values, neighbours in the map
        x = np.array([-0.5, 0.25, 0.2500001, 0.2500002, 3.0])[rng.integers(0, 5, d)]
    elif kind == "shared":          # weights that are already shared: runs of about a thousand equal ones
        x = rng.standard_normal(1 + d // 1000)[rng.integers(0, 1 + d // 1000, d)]
    elif kind == "binades":         # sixty binades, both signs
        x = np.ldexp(x, rng.integers(-30, 30, d))
    elif kind == "clusters":        # spikes that the cells of the map do not resolve
        x = rng.integers(-20, 20, d) + 1e-5 * x
    elif kind == "sorted":
        x = np.sort(x)
    elif kind == "constant":
        x = np.full(d, 0.37)
    return x.astype(dt)


def check(ws, ctx, w):
    dt = w.dtype.type
    plan = ws.Plan([0, w.shape[0]], TT[dt])
    s = torch.zeros(w.shape[0], dtype=TT[dt], device="cuda")
    plan.debug_sort(torch.from_numpy(w).cuda(), s)
    ctx.check(what="debug_sort")
    # the IEEE total order (-0 before +0) as signed integers
    b = w.view(UINT[dt])
    top = UINT[dt](1) << UINT[dt](8 * w.itemsize - 1)
    keys = np.sort(np.where(b & top, ~b, b | top))
    want = np.where(keys & top, keys ^ top, ~keys)
    assert np.array_equal(s.cpu().numpy().view(UINT[dt]), want)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("d", [2, 31, 2560, 4095, 4096, 4097, 5633, 6144, 6145, 40961])
def test_bin_edges(ws, ctx, d, dt):
    check(ws, ctx, draw("duplicates", d, dt))


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["narrow", "sparse", "few", "shared", "binades", "clusters", "sorted", "constant"])
def test_distributions(ws, ctx, kind, dt):
    check(ws, ctx, draw(kind, 300007, dt))


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["duplicates", "sparse", "clusters", "sorted"])
def test_two_passes(ws, ctx, kind, dt):
    check(ws, ctx, draw(kind, 512 * 2560 + 1 + 70001, dt))


def test_segments(ws, ctx):
    """One- and two-pass segments, ties and tiny ones side by side."""
    kinds = ["duplicates", "constant", "sparse", "few", "narrow", "clusters"]
    lens = [1600000, 5000, 70000, 2, 40000, 9001, 4097, 1500001]
    parts = [draw(kinds[i % len(kinds)], n, np.float32, seed=i) for i, n in enumerate(lens)]
    w = np.concatenate(parts)
    plan = ws.Plan(np.concatenate([[0], np.cumsum(lens)]), torch.float32)
    s = torch.zeros(w.shape[0], device="cuda")
    for _ in range(2):   # (a second call finds the first one's cursors and cells)
        plan.debug_sort(torch.from_numpy(w).cuda(), s)
        ctx.check(what="debug_sort")
        got = np.split(s.cpu().numpy(), np.cumsum(lens)[:-1])
        for g, p in zip(got, parts):
            assert np.array_equal(np.sort(g), g) and np.array_equal(np.sort(p), g)


def test_more_bins_than_16_bits_number(ws, ctx):
    """A segment of more than 65536 bins (their numbers take 32 bits), sorted and brought back to its order."""
    d = 65537 * 2560 + 12345
    g = torch.Generator(device="cuda").manual_seed(11)
    w = torch.randn(d, generator=g, device="cuda")
    w[::10] = w[1]
    want, order = torch.sort(w)
    plan = ws.Plan([0, d])
    s = torch.zeros_like(w)
    plan.debug_sort(w, s)
    ctx.check(what="debug_sort")
    assert torch.equal(s, want)
    out, ids, _ = plan.forward(w, torch.zeros(1, dtype=torch.float64, device="cuda"))
    ctx.check(what="prox")
    # lambda 0: equal weights are one cluster; a weight alone is its own value, the mean of several equal ones has
    # the four roundings of the FP32 value at most (it is not promised to be the weight itself)
    alone = torch.bincount(ids)[ids] == 1
    assert torch.equal(out[alone], w[alone])
    assert torch.all((out - w).abs() <= 2.0 ** -22 * w.abs())
    step = (ids[order][1:] - ids[order][:-1])
    assert torch.equal(step, (want[1:] != want[:-1]).int())


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["uniform", "one side", "with zeros", "tiny outliers", "two spikes"])
@pytest.mark.parametrize("d", [4097, 50000, 700001, 3000001])
def test_hard_edges_and_the_gap_around_zero(ws, ctx, dt, kind, d):
    """The map's ends (the parts of the smallest and the largest sample) and, in FP64, its closed gap
    around zero: magnitudes below the sampled ones, on both sides, zeros of both signs, denormals."""
    rng = np.random.default_rng(d)
    x = rng.uniform(-0.038, 0.038, d)
    if kind == "one side":
        x = np.abs(x) + 1.0
    elif kind == "with zeros":
        x[rng.random(d) < 0.01] = 0.0
        x[rng.random(d) < 0.01] *= -0.0
    elif kind == "tiny outliers":
        tiny = np.finfo(dt).smallest_subnormal
        x[:64] = np.arange(-32, 32) * float(tiny)
        x[64:70] = [1e30, -1e30, 1e-30, -1e-30, 3e-38, -3e-38]
        rng.shuffle(x)
    elif kind == "two spikes":
        x = np.where(x < 0, -1.0, 1.0) + 1e-6 * x
    check(ws, ctx, x.astype(dt))


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["cauchy", "lognormal", "negative lognormal", "one-sided cauchy", "tail and ties"])
@pytest.mark.parametrize("d", [4097, 20000, 300001])
def test_heavy_tails(ws, ctx, kind, d, dt):
    """Bins over many binades with most of their keys at the end next to zero."""
    rng = np.random.default_rng(d + 1)
    x = rng.standard_cauchy(d)
    if kind == "lognormal":
        x = np.exp(4 * rng.standard_normal(d))
    elif kind == "negative lognormal":
        x = -np.exp(4 * rng.standard_normal(d))
    elif kind == "one-sided cauchy":
        x = np.abs(x)
    elif kind == "tail and ties":
        x = np.where(rng.random(d) < 0.3, 1e-3, np.exp(5 * rng.standard_normal(d)))
    check(ws, ctx, x.astype(dt))
