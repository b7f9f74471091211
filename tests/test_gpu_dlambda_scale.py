"""d/d lambda of device-wide segments is as accurate as a sum of FP64 products: the error stays below a few
roundings of the sum of the magnitudes, whatever the exponents and wherever the largest gradient lies."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

from test_gpu_dlambda import TILE, cluster_ids, weights, ws  # noqa: F401  (ws: fixture)

pytestmark = pytest.mark.gpu


def run(ws, g, ids, dt):  # noqa: F811
    got = ws.prox_dlambda(torch.from_numpy(g).cuda().to(dt), torch.from_numpy(ids.astype(np.int32)).cuda())
    ws.Context.get().check(what="dlambda")
    return Fraction(got.item())


def check(got, g, ids):
    # per tile: products and sum within 2^-98 of its largest product, a conversion and a division; then the tiles'
    # sums one by one
    k, n = weights(ids), len(ids)
    terms = [Fraction(float(x)) * int(y) for x, y in zip(g, k)]
    want, mag = sum(terms, Fraction(0)) / (n - 1), sum(map(abs, terms), Fraction(0)) / (n - 1)
    assert abs(got - want) <= (math.ceil(n / TILE) + 4) * Fraction(2) ** -53 * mag


@pytest.mark.parametrize("dt,big", [(torch.float32, 70), (torch.float32, 120), (torch.float64, 70), (torch.float64, 900)])
@pytest.mark.parametrize("n", [4097, 2 * TILE + 1])
def test_huge_gradient_of_the_middle_cluster(ws, dt, big, n):  # noqa: F811
    """The middle cluster does not move with lambda: its gradient, however large, takes nothing from the others."""
    ids = np.arange(n)[::-1].copy()
    g = np.ones(n)
    g[: n // 3] = 3.0
    g[n // 2] = 2.0 ** big
    assert weights(ids)[n // 2] == 0
    check(run(ws, g, ids, dt), g, ids)


@pytest.mark.parametrize("dt,lo,hi", [(torch.float32, -140, 120), (torch.float32, -30, 0), (torch.float64, -1000, 900),
                                      (torch.float64, -40, 0), (torch.float64, -100, 0)])
@pytest.mark.parametrize("kind", ["distinct", "crowd", "pairs"])
def test_exponents(ws, kind, dt, lo, hi):  # noqa: F811
    rng = np.random.default_rng(11)
    n = 3 * TILE + 5
    ids = cluster_ids(kind, n, rng)
    g = np.ldexp(rng.standard_normal(n), rng.integers(lo, hi + 1, n))
    g = g.astype(np.float32).astype(np.float64) if dt == torch.float32 else g
    check(run(ws, g, ids, dt), g, ids)


@pytest.mark.parametrize("dt,small", [(torch.float32, -45), (torch.float64, -40)])
def test_largest_gradients_have_the_smallest_weights(ws, dt, small):  # noqa: F811
    """The weights go up to the segment's length: small gradients count as much as a large one of weight 1."""
    n = 1 << 17
    ids = np.arange(n)
    rng = np.random.default_rng(13)
    g = np.ldexp(rng.standard_normal(n), small)
    g = g.astype(np.float32).astype(np.float64) if dt == torch.float32 else g
    g[np.abs(weights(ids)) == 1] = 1.0
    check(run(ws, g, ids, dt), g, ids)
