"""d/d lambda against sums of integers: cluster sizes that meet in one tile (counted
through shared memory), distinct ones, several segments with slot counts that are no
multiple of four; infinities and NaN; gradients over a wide range of exponents."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

TILE, SAMPLE = 6144, 512


@pytest.fixture(scope="module")
def ws():
    from paper_2311_03096_gb300 import ws as m

    return m


def cluster_ids(kind, n, rng):
    if kind == "one":
        return np.zeros(n, np.int64)
    if kind == "distinct":
        return rng.permutation(n)
    if kind == "few":
        return rng.integers(0, min(7, n), n)
    if kind == "pairs":                     # about the number of meetings that selects the table
        return rng.integers(0, min(2000, n), n)
    if kind == "crowd":                     # the table full of short clusters around a huge one
        c = max(n // 3, 1)
        return np.where(rng.random(n) < 0.5, c // 2, rng.integers(0, c, n))
    if kind == "neighbours":
        return np.arange(n) // 3
    raise ValueError(kind)


def weights(ids):
    """len - 2 start - size of every element's cluster."""
    n = len(ids)
    size = np.bincount(ids, minlength=n).astype(np.int64)
    start = np.cumsum(size) - size
    return (n - 2 * start - size)[ids]


def close(got, g, ids):
    # one CTA's sum is an integer, converted and divided (three roundings); the tiles are added one by one in FP64
    k = weights(ids)
    n = len(ids)
    want = Fraction(int(np.sum(g * k)), n - 1)
    mag = int(np.sum(np.abs(g * k))) / (n - 1)
    assert abs(Fraction(float(got)) - want) <= Fraction((math.ceil(n / TILE) + 4) * 2.0 ** -53 * mag)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("kind", ["one", "distinct", "few", "pairs", "crowd", "neighbours"])
@pytest.mark.parametrize("n", [4097, TILE + SAMPLE - 1, 4 * TILE, 1000003])
def test_counts(ws, dt, kind, n):
    rng = np.random.default_rng(n)
    ids = cluster_ids(kind, n, rng)
    g = rng.integers(-1024, 1024, n)
    got = ws.prox_dlambda(torch.from_numpy(g).cuda().to(dt), torch.from_numpy(ids.astype(np.int32)).cuda())
    ws.Context.get().check(what="dlambda")
    close(got.item(), g, ids)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_segments(ws, dt):
    rng = np.random.default_rng(3)
    lens = [5000, 17, 4099, 70001, 4096, 8193]
    offs = np.concatenate([[0], np.cumsum(lens)])
    ids = [cluster_ids(k, n, rng) for k, n in zip(["crowd", "few", "distinct", "pairs", "one", "neighbours"], lens)]
    g = rng.integers(-1024, 1024, int(offs[-1]))
    plan = ws.Plan(offs, dtype=dt)
    got = plan.dlambda(torch.from_numpy(g).cuda().to(dt), torch.from_numpy(np.concatenate(ids).astype(np.int32)).cuda())
    ws.Context.get().check(what="dlambda")
    for s, i in enumerate(ids):
        close(got[s].item(), g[offs[s]:offs[s + 1]], i)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("bad", [math.inf, -math.inf, math.nan])
def test_not_finite(ws, dt, bad):
    rng = np.random.default_rng(4)
    n = 9001
    ids = cluster_ids("few", n, rng)
    g = rng.standard_normal(n)
    at = int(np.nonzero(weights(ids))[0][100])
    g[at] = bad
    got = ws.prox_dlambda(torch.from_numpy(g).cuda().to(dt), torch.from_numpy(ids.astype(np.int32)).cuda()).item()
    want = bad * weights(ids)[at]
    assert math.isnan(got) if math.isnan(want) else got == want


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_wide_exponents(ws, dt):
    """Values far below a tile's largest one keep at least 62 bits under its top, which an FP64 sum does not."""
    rng = np.random.default_rng(6)
    n = 3 * TILE + 5
    ids = cluster_ids("crowd", n, rng)
    lo, hi = (-140, 120) if dt == torch.float32 else (-1000, 900)
    g = np.ldexp(rng.standard_normal(n), rng.integers(lo, hi, n))
    g = g.astype(np.float32).astype(np.float64) if dt == torch.float32 else g
    got = ws.prox_dlambda(torch.from_numpy(g).cuda().to(dt), torch.from_numpy(ids.astype(np.int32)).cuda()).item()
    k = weights(ids)
    want = sum((Fraction(float(x)) * int(y) for x, y in zip(g, k)), Fraction(0)) / (n - 1)
    mag = sum((abs(Fraction(float(x)) * int(y)) for x, y in zip(g, k)), Fraction(0)) / (n - 1)
    # (four tiles; a dropped part is below 2^-61 of its tile's largest value, times n elements of weight n at most)
    top = Fraction(float(np.abs(g).max()))
    assert abs(Fraction(got) - want) <= 8 * Fraction(2) ** -53 * mag + n * n * top * Fraction(2) ** -61 / (n - 1)
