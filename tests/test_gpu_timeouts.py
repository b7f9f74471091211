"""Waits of the sort's grid barriers that give up, in the plan kernel and (with the plan's short
waits just fitting the limit) in the sort of oversize bins: the call ends with WS_ERR_TIMEOUT or
with the right result, and the next call without a limit is right."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
LIMITS = [1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 48, 64, 80, 96, 128, 192, 256, 512, 1024, 4096]


@pytest.fixture
def ctx():
    from paper_2311_03096_gb300 import ws

    c = ws.Context.get()
    yield c
    c.set_spin_limit(0)
    c.status()


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("share", [0.02, 0.5, 1.0])
def test_waits_that_give_up(ctx, dt, share):
    from paper_2311_03096_gb300 import ws

    d = 1 << 20
    rng = np.random.default_rng(8)
    x = rng.standard_normal(d)
    x[rng.random(d) < share] = 0.25
    w = torch.from_numpy(x).cuda().to(dt)
    prec = "fp64" if dt == torch.float64 else "fp32comp"
    calls = [lambda: ws.prox(w, 0.01, prec), lambda: ws.R(w)]
    want = [f() for f in calls]
    ctx.check(what="reference")
    seen = set()
    for limit in LIMITS:
        ctx.set_spin_limit(limit)
        for f, r in zip(calls, want):
            got = f()
            st = ctx.status()
            seen.add(st)
            assert st in (ws.WS_OK, ws.WS_ERR_TIMEOUT)
            if st == ws.WS_OK:
                assert all(torch.equal(a, b) for a, b in zip(got, r))
    assert ws.WS_ERR_TIMEOUT in seen
    ctx.set_spin_limit(0)
    for f, r in zip(calls, want):
        got = f()
        ctx.check(what="after the timeouts")
        assert all(torch.equal(a, b) for a, b in zip(got, r))
