"""Junctions whose bridge drops hundreds to thousands of a tile hull's vertices (the
tails of a distribution around one large cluster), on either side, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from parity import compare_segment  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,prec,tol", [(np.float32, "fp32comp", 1e-5), (np.float64, "fp64", 1e-10)])
@pytest.mark.parametrize("kind", ["normal", "left", "right", "plateau"])
@pytest.mark.parametrize("d", [8192, 8193, 50000])
@pytest.mark.parametrize("lam", [3.0, 10.0, 30.0])
def test_against_oracle(dt, prec, tol, kind, d, lam):
    from paper_2311_03096_gb300 import ws

    rng = np.random.default_rng(d)
    w = rng.standard_normal(d)
    if kind == "left":            # one long tail
        w = -np.abs(w) ** 3
    elif kind == "right":
        w = np.abs(w) ** 3
    elif kind == "plateau":       # most of the weights in a narrow middle
        w = np.where(rng.random(d) < 0.9, 1e-3 * w, 8 * w)
    w = w.astype(dt)
    out, ids, nc = ws.prox(torch.from_numpy(w).cuda(), lam, prec)
    ws.Context.get().check(what="prox")
    ref = oracle.prox(w, lam, return_perm=True)
    compare_segment(w, lam, out.cpu().numpy(), ids.cpu().numpy(), int(nc.item()), tol, ref=ref)
