"""The fp32 kernel (scores, test and routing of a row tile in one kernel) at its edges: both row-tile
heights, partial tiles, key chunks around the 256 / 512-chunk passes, the largest strip, rows that
see fewer chunks than their route is wide, and agreement with the two-pass path."""
import pytest
import torch

import parity
from paper_2609_07306_b200 import workload as W
from paper_2609_07306_b200.ledger import RouteLedger, config_from_workload, device_tensor

pytestmark = pytest.mark.gpu


def _w(heads, n_q, n_k, d, k, m, r, causal, **kw):
    return W.RouteWorkload("f32_edge", 1, heads, n_q, n_k, d, k, m, r, layers=3, anchor_every=100, dtype=W.DTYPE_F32,
                           centroids=8, rho=0.2, causal=causal, seed=31, **kw)


@pytest.mark.parametrize("heads,n_q,n_k,d,k,m,r,causal", [
    (1, 1, 1, 64, 1, 0, 0, False), (2, 17, 33, 64, 6, 4, 3, False), (1, 130, 257, 128, 12, 8, 8, True),
    (2, 40, 513, 64, 16, 8, 5, False), (9, 601, 130, 64, 9, 7, 6, True), (1, 24, 4096, 128, 40, 24, 8, False)])
def test_f32_kernel_parity(heads, n_q, n_k, d, k, m, r, causal):
    rep = parity.run_teacher_forced(_w(heads, n_q, n_k, d, k, m, r, causal, global_sentinels=3 if k > 1 else 0))
    parity.assert_clean(rep)


def test_f32_kernel_equals_the_two_pass_anchor():
    w = _w(3, 200, 333, 64, 12, 8, 8, True, causal_offset=100)
    q, k = W.generate(w, layers=1)
    leds = [RouteLedger(config_from_workload(w, two_pass=t)) for t in (False, True)]
    for led in leds:
        led.route_anchor(device_tensor(q[0]), device_tensor(k[0]), 0)
    torch.cuda.synchronize()
    for name in ("routes", "sentinels", "kth_score", "margin", "ages", "flags"):
        assert torch.equal(getattr(leds[0], name), getattr(leds[1], name)), name
    for led in leds:
        led.close()
