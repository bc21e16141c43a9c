"""A wait that expires while the routing kernel decides about a relay's rows: the four warps that share a quarter of the
rows must go the same way whatever each of them could see of the abort flag, or some would wait at a barrier that the
others never reach.  A test hook (debug bit 9) raises the flag in one warp right after the decision."""
import pytest
import torch

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200 import workload as W
from paper_2609_07306_b200.ledger import RouteLedger, config_from_workload, device_tensor

pytestmark = pytest.mark.gpu


# (rho 0: every row passes the test, the other way out of the decision)
@pytest.mark.parametrize("rho", [0.0, 0.3])
@pytest.mark.parametrize("heads", [2, 40])
def test_quarter_agrees_when_a_wait_expires_at_the_decision(heads, rho):
    w = W.moderate().replace(heads=heads, rho=rho)
    q, k = W.generate(w, layers=2)
    dq, dk = [device_tensor(x) for x in q], [device_tensor(x) for x in k]
    cfg = config_from_workload(w)
    cfg.debug_outputs |= 1 << 9
    led, ref = RouteLedger(cfg), RouteLedger(config_from_workload(w))
    for x in (led, ref):
        x.route_anchor(dq[0], dk[0], 0)
    assert led.status() == 0
    for x in (led, ref):
        x.route_relay(dq[1], dk[1], 1)
    with pytest.raises(B.RouteRelayError) as ei:
        led.status()
    assert ei.value.code == B.RR_ERR_TIMEOUT and ref.status() == 0
    # the first CTA holds the last row tile of the first problem; every other row is as if nothing had happened
    free = torch.ones(w.rows, dtype=torch.bool, device="cuda")
    free[w.n_q - 128:w.n_q] = False
    for f in ("flags", "routes", "sentinels", "kth_score"):
        assert torch.equal(getattr(led, f)[free], getattr(ref, f)[free]), f
    # the hook fires once per ledger
    for x in (led, ref):
        x.reset()
        for l in range(2):
            (x.route_relay if l else x.route_anchor)(dq[l], dk[l], l)
    assert led.status() == 0
    for f in ("flags", "routes", "sentinels", "ages", "refresh_count"):
        assert torch.equal(getattr(led, f), getattr(ref, f)), f
    led.close(); ref.close()
