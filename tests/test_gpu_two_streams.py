"""Device-wide calls of two plans that overlap on two streams: each has grids that wait for all of their
CTAs, so the two must not take the device from each other half by half."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    from paper_2311_03096_gb300 import ws

    return ws.Context.get()


@pytest.mark.parametrize("sizes", [(1 << 24, 1 << 24), (300007, 5000001), (41000, 1 << 22)])
def test_two_plans_on_two_streams(ctx, sizes):
    from paper_2311_03096_gb300 import ws

    ws_, plans, want = [], [], []
    lam = torch.full((1,), 0.05, dtype=torch.float64, device="cuda")
    for i, d in enumerate(sizes):
        ws_.append(torch.randn(d, generator=torch.Generator(device="cuda").manual_seed(30 + i), device="cuda"))
        plans.append(ws.Plan([0, d]))
        want.append(plans[i].forward(ws_[i], lam))
    ctx.check(what="one after the other")
    streams = [torch.cuda.Stream() for _ in sizes]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(10):
        for i, s in enumerate(streams):
            with torch.cuda.stream(s):
                got[i].append(plans[i].forward(ws_[i], lam))
    torch.cuda.synchronize()
    ctx.check(what="side by side")
    for i in range(2):
        for r in got[i]:
            assert all(torch.equal(a, b) for a, b in zip(r, want[i]))
