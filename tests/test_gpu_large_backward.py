"""The device-wide backward: every mean against sums of integers, at the edges of
its bins and moves, and with clusters that split a bin, fill whole tiles or
crowd a warp."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

BIN, FAN, TILE, PIECE = 2048, 512, 6144, 16384   # slots per bin, bins per move, elements per tile, pairs per CTA


@pytest.fixture(scope="module")
def ws():
    from paper_2311_03096_gb300 import ws as m

    return m


def cluster_ids(kind, n, rng):
    if kind == "one":                       # every tile adds its sum once
        return np.zeros(n, np.int64)
    if kind == "distinct":
        return rng.permutation(n)
    if kind == "few":                       # bins split over many CTAs
        return rng.integers(0, min(5, n), n)
    if kind == "last":                      # one bin, the last slots of the segment
        return n - 1 - rng.integers(0, min(n, 700), n)
    if kind == "crowd":                     # one cluster of half the elements, short ones around it
        c = max(n // 3, 1)
        return np.where(rng.random(n) < 0.5, c // 2, rng.integers(0, c, n))
    if kind == "blocks":                    # tiles of one cluster beside mixed ones, of the same bins
        ids = rng.integers(0, max(n // 7, 1), n)
        for a in range(0, n, 3 * TILE):
            ids[a:a + TILE] = 3 if (a // TILE) % 2 else n // 9
        return ids
    raise ValueError(kind)


def check(got, g, ids, n):
    # sums of integers below 2^20 are exact in int64; FP32: a rounding of the sum, one of the count, a division and
    # the scaling; FP64: an FP32 remainder quotient (2^-42)
    s = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, ids.long(), g.long())
    c = torch.bincount(ids.long(), minlength=n).clamp_(min=1)
    want = (s.double() / c.double())[ids.long()]
    rel = 4 * 2.0 ** -24 if g.dtype == torch.float32 else 2.0 ** -41
    assert torch.all((got.double() - want).abs() <= rel * want.abs())


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("kind", ["one", "distinct", "few", "last", "crowd", "blocks"])
@pytest.mark.parametrize("n", [4097, TILE + 1, 5 * BIN - 1, 7 * PIECE + 1, BIN * FAN, BIN * FAN + 1, 3000017])
def test_means(ws, dt, kind, n):
    rng = np.random.default_rng(n)
    ids = torch.from_numpy(cluster_ids(kind, n, rng).astype(np.int32)).cuda()
    g = torch.from_numpy(rng.integers(-2 ** 20, 2 ** 20, n)).cuda().to(dt)
    got = ws.prox_backward(g, ids)
    ws.Context.get().check(what="backward")
    check(got, g, ids, n)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_many_bins(ws, dt):
    """More bins than the shared-memory counts hold, over segments of both moves."""
    rng = np.random.default_rng(5)
    lens = [31000003, 5000, 17, 1048577, 2600000]
    offs = np.concatenate([[0], np.cumsum(lens)])
    plan = ws.Plan(offs, dtype=dt)
    ids = np.concatenate([cluster_ids(k, n, rng) for k, n in zip(["distinct", "crowd", "few", "blocks", "one"], lens)])
    ids = torch.from_numpy(ids.astype(np.int32)).cuda()
    g = torch.from_numpy(rng.integers(-2 ** 20, 2 ** 20, int(offs[-1]))).cuda().to(dt)
    got = plan.backward(g, ids)
    ws.Context.get().check(what="backward")
    for a, b in zip(offs[:-1], offs[1:]):
        check(got[a:b], g[a:b], ids[a:b], b - a)


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_wide_exponents(ws, dt):
    """Limbs of every height with carries through all of them: +-2^k pairs that
    cancel exactly beside an integer per cluster, in bins large enough to be normalised."""
    rng = np.random.default_rng(9)
    m, clusters = 40000, 900
    ids = rng.integers(0, clusters, m)
    small = rng.integers(-2 ** 20, 2 ** 20, m).astype(np.float64)
    big = np.ldexp(1.0, rng.integers(20, 60 if dt == torch.float32 else 40, m))
    g = np.concatenate([small, big, -big])
    idc = np.concatenate([ids, ids, ids])
    p = rng.permutation(3 * m)
    g, idc = g[p], idc[p]
    gt = torch.from_numpy(g).cuda().to(dt)
    it = torch.from_numpy(idc.astype(np.int32)).cuda()
    got = ws.prox_backward(gt, it)
    ws.Context.get().check(what="backward")
    s = np.bincount(ids, weights=small, minlength=clusters)      # (exact: integers below 2^53)
    want = torch.from_numpy((s / np.maximum(np.bincount(idc, minlength=clusters), 1))[idc]).cuda()
    rel = 4 * 2.0 ** -24 if dt == torch.float32 else 2.0 ** -41
    assert torch.all((got.double() - want).abs() <= rel * want.abs())
