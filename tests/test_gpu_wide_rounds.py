"""Segments and tiles whose prefix sums need 128 bits: the Imminent Collisions
rounds against the tree of merges (round cap 0), bit for bit, at the edges of the
lanes' chunks, over spreads of exponents, ties and clusters of every size; a cap
of 3 lets some rounds give up."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    from paper_2311_03096_gb300 import ws

    c = ws.Context.get(0)
    c.set_ic_cap(-1)
    yield c
    c.set_ic_cap(-1)


def vector(kind, n, dt, rng):
    w = rng.standard_normal(n)
    if kind == "wide":
        w = np.ldexp(w, rng.integers(-60, 60, n))
    elif kind == "ties":          # half of the neighbours equal, the others one unit apart
        w = np.sort(rng.integers(0, n // 2 + 1, n)) * 2.0 ** -20 + np.ldexp(1.0, rng.integers(-50, 3, n)) * (rng.random(n) < 0.01)
    elif kind == "lattice":       # exact ties of the hull test: equal steps
        w = np.arange(n) * 2.0 ** -8 - 3.0
        w[: n // 8] = np.ldexp(1.0, -40)
    return w.astype(dt)


@pytest.mark.parametrize("dt", [np.float64, np.float32])
@pytest.mark.parametrize("kind", ["normal", "wide", "ties", "lattice"])
@pytest.mark.parametrize("n", [2, 15, 17, 33, 513, 4080, 4081, 4096, 4097, 3 * 4096 + 17])
def test_rounds_match_merges(ctx, dt, kind, n):
    from paper_2311_03096_gb300 import ws

    w = torch.from_numpy(vector(kind, n, dt, np.random.default_rng(n))).cuda()
    prec = "fp64" if dt == np.float64 else "fp32comp"
    for lam in (0.0, 1e-3, 0.1, 1.0, (n - 1) / 2 * 2.0 ** -8, 30.0):
        ctx.set_ic_cap(0)
        want = ws.prox(w, lam, prec)
        ctx.check(what="merges")
        for cap in (3, -1):
            ctx.set_ic_cap(cap)
            got = ws.prox(w, lam, prec)
            ctx.check(what="rounds")
            for a, b in zip(got, want):
                assert torch.equal(a, b)
