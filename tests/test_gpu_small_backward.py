"""The one-CTA backward's limb sums against exact rational sums: values over the
whole exponent range, cancellations, one cluster of the largest segment (the
limbs' headroom), sizes around the CTA's thread count."""
import math
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ws():
    from paper_2311_03096_gb300 import ws as m

    return m


def grads(kind, n, dt, rng):
    g = rng.standard_normal(n)
    if kind == "wide":              # from denormals to near the largest value
        lo, hi = (-149, 120) if dt == np.float32 else (-1074, 1000)
        g = np.ldexp(g, rng.integers(lo, hi, n))
    elif kind == "cancel":          # pairs that cancel to a small remainder
        g = np.where(np.arange(n) % 2 == 0, 2.0 ** 40, -2.0 ** 40) + np.round(g * 8) / 8
    elif kind == "largest":         # every limb of every value full, one sign
        g = np.full(n, 1.0 - 2.0 ** (-24 if dt == np.float32 else -53))
    elif kind == "zeros":
        g = np.zeros(n)
    return g.astype(dt)


@pytest.mark.parametrize("dt", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["normal", "wide", "cancel", "largest", "zeros"])
@pytest.mark.parametrize("n,clusters", [(1, 1), (31, 5), (511, 511), (513, 40), (4095, 3), (4096, 1), (4096, 4096)])
def test_limb_sums(ws, dt, kind, n, clusters):
    rng = np.random.default_rng(n + clusters)
    g = grads(kind, n, dt, rng)
    ids = rng.permutation(np.concatenate([np.arange(clusters), rng.integers(0, clusters, n - clusters)])).astype(np.int32)
    got = ws.prox_backward(torch.from_numpy(g).cuda(), torch.from_numpy(ids).cuda())
    ws.Context.get().check(what="backward")
    got = got.cpu().numpy()
    top = math.frexp(float(np.abs(g).max()))[1] - 1 if np.any(g) else 0
    # FP32: two conversions, a division and a rounding; FP64: an FP32 remainder quotient (2^-42).
    # Values more than 71 (42) binades below the largest keep their top bits only.
    rel = Fraction(4, 2 ** 24) if dt == np.float32 else Fraction(2, 2 ** 42)
    cut = Fraction(2) ** (top - (71 + 23 if dt == np.float32 else 42 + 52))
    tiny = Fraction(2) ** (-149 if dt == np.float32 else -1074)
    for c in range(clusters):
        at = np.nonzero(ids == c)[0]
        mean = sum((Fraction(float(x)) for x in g[at]), Fraction(0)) / len(at)
        vals = got[at]
        assert np.all(vals == vals[0])
        assert abs(Fraction(float(vals[0])) - mean) <= rel * abs(mean) + cut + tiny
