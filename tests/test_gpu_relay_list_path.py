"""A relay whose test is a kernel of its own, with the list between it and the routing kernel (debug bit 10: on any grid),
and the test inside the routing kernel with every number of rows per CTA, held against it bit for bit; the lines between
the column capacities of the routing kernel with four threads per row, against the two-pass path."""
import pytest
import torch

import parity
from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200 import workload as W
from paper_2609_07306_b200.ledger import RouteLedger, config_from_workload, device_tensor

pytestmark = pytest.mark.gpu

LIST = 1 << 10
FIELDS = ("routes", "sentinels", "ages", "kth_score", "margin", "flags", "alpha", "beta", "problem_offsets", "refresh_count",
          "counters", "force_state")


def _bits(x):
    return x.view(torch.int32) if x.dtype == torch.float32 else x


def _config(w, bits=0, **kw):
    cfg = config_from_workload(w, **kw)
    cfg.debug_outputs |= bits
    return cfg


def test_rescoring_kernel_gives_up_and_recovers():
    w = W.moderate().replace(heads=2)
    q, k = W.generate(w, layers=2)
    dq, dk = [device_tensor(x) for x in q], [device_tensor(x) for x in k]
    led, ref = RouteLedger(_config(w, LIST, forced_timeouts=2)), RouteLedger(_config(w, LIST))
    for x in (led, ref):
        x.route_anchor(dq[0], dk[0], 0)
        x.route_relay(dq[1], dk[1], 1)
    with pytest.raises(B.RouteRelayError) as ei:
        led.status()
    assert ei.value.code == B.RR_ERR_TIMEOUT and ref.status() == 0
    free = torch.ones(w.rows, dtype=torch.bool, device="cuda")
    free[w.n_q - 128:w.n_q] = False                          # the first CTA's rows
    assert torch.equal(led.flags[free], ref.flags[free])
    for x in (led, ref):
        x.reset()
        x.route_anchor(dq[0], dk[0], 0)
        x.route_relay(dq[1], dk[1], 1)
    assert led.status() == 0
    for f in FIELDS:
        assert torch.equal(_bits(getattr(led, f)), _bits(getattr(ref, f))), f
    led.close(); ref.close()


# (widths whose ledger rows do and do not split into 16 bytes, no sentinels, more loads than a batch)
@pytest.mark.parametrize("n_q,n_k,d,k,m,r,causal", [
    (1, 40, 64, 1, 0, 1, False), (31, 65, 128, 4, 4, 4, True), (33, 97, 64, 5, 3, 0, True),
    (97, 300, 128, 3, 0, 0, False), (129, 333, 64, 64, 32, 31, False), (160, 2048, 128, 9, 1, 8, True),
])
def test_ledger_rows_of_all_widths_with_a_list(monkeypatch, n_q, n_k, d, k, m, r, causal):
    monkeypatch.setattr(parity, "config_from_workload", lambda *a, **kw: _config(a[0], LIST, **kw))
    w = W.RouteWorkload("edge", 1, 3, n_q, n_k, d, k, m, r, layers=4, anchor_every=100, dtype=W.DTYPE_BF16,
                        centroids=10, rho=0.2, causal=causal, causal_offset=max(0, n_k - n_q), seed=8)
    parity.assert_clean(parity.run_teacher_forced(w))


# 32 rows per CTA; 64; 128; the most tiles that the test inside the routing kernel takes; forced anchors in both
@pytest.mark.parametrize("P,n_q,n_k,d,k,m,r,extra", [
    (2, 300, 256, 128, 32, 16, 8, dict(force_permille=300, force_max_run=2)),
    (8, 256, 256, 128, 16, 8, 8, dict(force_permille=300, force_max_run=2)),
    (15, 389, 500, 64, 20, 10, 7, dict(causal_offset=111)),
    (40, 160, 300, 128, 50, 30, 16, dict(force_permille=300, force_max_run=2)),
    (49, 300, 200, 64, 12, 4, 5, dict(causal=0)),
    (74, 129, 400, 128, 40, 16, 16, dict(causal_offset=271, gamma=0.01)),
    (148, 100, 128, 64, 24, 12, 12, {}),
    (1, 2000, 700, 128, 40, 8, 0, dict(global_sentinels=3)),
])
@pytest.mark.parametrize("rho", [0.02, 0.3])
def test_test_in_the_routing_kernel_equals_the_list(P, n_q, n_k, d, k, m, r, extra, rho):
    g = torch.Generator(device="cuda").manual_seed(P + n_q)
    cfg = dict(batch=1, heads=P, n_q=n_q, n_k=n_k, d=d, k=k, m=m, r=r, dtype=B.RR_BF16, causal=1, causal_offset=0, seed=3)
    cfg.update(extra)
    rnd = lambda n: torch.randn((P, n, d), generator=g, device="cuda") * d ** -0.5
    q, kk = rnd(n_q), rnd(n_k)
    inside, lists = RouteLedger(B.rr_config(**cfg)), RouteLedger(B.rr_config(debug_outputs=LIST, **cfg))
    launches = []
    for l in range(7):
        for led in (inside, lists):
            before = B.rr_kernel_launch_count()
            (led.route_anchor if l == 0 else led.route_relay)(q.bfloat16(), kk.bfloat16(), l)
            launches.append(B.rr_kernel_launch_count() - before)
        assert inside.status() == 0 and lists.status() == 0
        for f in FIELDS:
            assert torch.equal(_bits(getattr(inside, f)), _bits(getattr(lists, f))), (f, l)
        n = int(inside.refresh_count.item())
        assert torch.equal(inside.refresh_rows[:n], lists.refresh_rows[:n]), l
        q, kk = ((1 - rho * rho) ** 0.5 * x + rho * rnd(x.shape[1]) for x in (q, kk))
    assert launches[3] == launches[2] + 1                    # (the two differ in what they launch)
    if "force_permille" in extra and rho == 0.3:
        assert inside.force_state[4].item() > 0              # (forced calls were among them)
    inside.close(); lists.close()


# (key chunks at the upper end of each line of the rule, and one beyond; the last kept width of a column and the next)
@pytest.mark.parametrize("n_k,d,keep", [
    (200, 128, 40), (256, 128, 70), (256, 64, 76), (256, 128, 88), (257, 128, 66), (320, 64, 72), (320, 128, 74),
    (320, 128, 86), (321, 64, 62), (512, 64, 68), (512, 128, 76), (512, 128, 88), (513, 128, 58), (1024, 64, 64),
    (1024, 128, 70), (1024, 128, 84), (1536, 128, 56), (1536, 64, 62), (1536, 64, 70), (1536, 128, 82), (2048, 64, 56),
    (2048, 128, 68), (2048, 128, 82), (2049, 128, 48), (2049, 64, 66), (2500, 128, 80),
])
def test_lines_between_the_columns(n_k, d, keep):
    g = torch.Generator(device="cuda").manual_seed(keep + n_k)
    for kept in (keep, keep + 1):
        m = kept // 3
        w = W.RouteWorkload("line", 1, 2, 140, n_k, d, kept - m, m, 8, layers=2, anchor_every=100, dtype=W.DTYPE_BF16,
                            centroids=12, rho=0.2, causal=False, seed=9)
        q, k = (torch.randn((2, n, d), generator=g, device="cuda").bfloat16() for n in (140, n_k))
        got = []
        for two_pass in (False, True):
            led = RouteLedger(config_from_workload(w, two_pass=two_pass))
            led.route_anchor(q, k, 3)
            assert led.status() == 0
            got.append([led.routes.sort(1).values, led.sentinels[:, :m].sort(1).values, led.sentinels[:, m:].clone(),
                        _bits(led.kth_score).clone(), _bits(led.margin).clone()])
            led.close()
        assert all(torch.equal(a, b) for a, b in zip(*got)), kept
