"""The forward of the device-wide path on the inputs that the sort finds hard: bins that span
more key bits than a word keeps, with ties among them; heavy ties; distributions that the
sampled map does not resolve; with one and two partition passes to undo."""
import numpy as np
import pytest
import torch

from parity import compare_segment
from test_gpu_sort import TT, draw

pytestmark = pytest.mark.gpu
ONE, TWO = 300007, 512 * 2560 + 70002   # elements that take one partition pass, and two
TOL = {np.float32: 1e-5, np.float64: 1e-12}


@pytest.fixture(scope="module")
def ws():
    from paper_2311_03096_gb300 import ws as m

    return m


def with_zeros(d, n, dt, seed):
    """Weights around zero, n of them exact zeros of both signs."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-0.04, 0.04, d).astype(dt)
    x[rng.choice(d, n, replace=False)] = np.where(rng.random(n) < 0.5, 0.0, -0.0)
    return x


def forward(ws, w, lam):
    dt = w.dtype.type
    out, ids, nc = ws.prox(torch.from_numpy(w).cuda(), lam, "fp64" if dt == np.float64 else "fp32comp")
    ws.Context.get().check(what="prox")
    return out, ids, nc


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("d", [5000, 40961, TWO])
@pytest.mark.parametrize("n", [31, 33, 257, 2000])
def test_zeros_in_a_wide_bin(ws, dt, d, n):
    """A bin across zero spans nearly every key bit: its words leave some out, and the zeros are a
    run with equal top bits, above or below the length that one thread orders."""
    w = with_zeros(d, n, dt, seed=d + n)
    lam = 1e-3
    out, ids, nc = forward(ws, w, lam)
    compare_segment(w, lam, out.cpu().numpy(), ids.cpu().numpy(), nc.item(), TOL[dt])
    x = torch.from_numpy(w).cuda()
    for _ in range(100):
        o2, i2, n2 = ws.prox(x, lam, "fp64" if dt == np.float64 else "fp32comp")
        assert torch.equal(o2, out) and torch.equal(i2, ids) and torch.equal(n2, nc)
    ws.Context.get().check(what="prox")


def check_lambda_zero(ws, w):
    """lambda 0: the clusters are the different values, in their order.  (Weights within two units
    of the fixed point, 2^-56 of the largest, may share one.)"""
    out, ids, nc = (t.cpu().numpy() for t in forward(ws, w, 0.0))
    order = np.argsort(w, kind="stable")
    xs, g, v = w[order].astype(np.longdouble), ids[order], out[order].astype(np.longdouble)
    step, gap, top = np.diff(g), np.diff(xs), np.abs(xs).max()
    unit = top * np.longdouble(2) ** -56
    assert g[0] == 0 and int(nc[0]) == int(g[-1]) + 1
    assert np.all((step == 0) | (step == 1)) and np.all(step[gap == 0] == 0) and np.all(step[gap >= unit] == 1)
    # a value is the mean of its cluster: four roundings of the FP32 value, 2^-42 and two roundings of FP64's
    eps = 2.0 ** -22 if w.dtype == np.float32 else 2.0 ** -41
    assert np.all(np.abs(v - xs) <= eps * np.abs(xs) + 4 * unit * np.bincount(g)[g])


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("d", [ONE, TWO])
@pytest.mark.parametrize("kind", ["duplicates", "narrow", "sparse", "few", "shared", "binades", "clusters", "sorted",
                                  "constant"])
def test_distributions(ws, kind, d, dt):
    check_lambda_zero(ws, draw(kind, d, dt))


@pytest.mark.parametrize("d", [(1 << 19) * 2560 + 12345, (1 << 19) * 3000 + 77])
def test_bins_at_19_bits(ws, d):
    """Segments of 2^19 bins and of more, with a tie of about a million copies: at lambda 0 the ids number the
    values in their order."""
    ctx = ws.Context.get()
    ctx.set_small_max(-1)   # (drops the cached plans)
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 180e9:
        pytest.skip("needs 180 GB")
    w = torch.randn(d, generator=torch.Generator(device="cuda").manual_seed(12), device="cuda")
    w[w.abs() < 2.0 ** -10] = 2.0 ** -10   # (no value loses bits in the fixed point)
    plan = ws.Plan([0, d])
    out, ids, nc = plan.forward(w, torch.zeros(1, dtype=torch.float64, device="cuda"))
    ctx.check(what="prox")
    c = int(nc.item())
    assert int(ids.min()) == 0 and int(ids.max()) == c - 1
    value = torch.full((c,), float("nan"), device="cuda")
    for i in range(0, d, 1 << 28):
        value[ids[i:i + (1 << 28)]] = w[i:i + (1 << 28)]
    assert bool(torch.all(value[1:] > value[:-1]))
    for i in range(0, d, 1 << 28):
        x = w[i:i + (1 << 28)]
        assert torch.equal(value[ids[i:i + (1 << 28)]], x)
        assert bool(torch.all((out[i:i + (1 << 28)] - x).abs() <= 2.0 ** -22 * x.abs()))
