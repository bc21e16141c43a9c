"""One relay call captured as a graph and replayed: a call's refresh list, offsets and ages come from this call's flags and
not from what an earlier call has left in the scratch, however often and at whatever parity the same call runs."""
import pytest
import torch

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200.ledger import RouteLedger

pytestmark = pytest.mark.gpu

FIELDS = ("routes", "sentinels", "ages", "kth_score", "margin", "flags", "problem_offsets", "refresh_count")


# (tests inside the routing kernel with 32, 64 and 128 rows per CTA, ragged problems; a test kernel of its own; fp32 CTAs
# of 8 and 16 rows)
@pytest.mark.parametrize("P,n_q,n_k,d,dtype,extra", [
    (3, 300, 256, 128, torch.bfloat16, {}),
    (15, 389, 500, 64, torch.bfloat16, {}),
    (70, 150, 130, 64, torch.bfloat16, dict(causal=0)),
    (80, 200, 256, 128, torch.bfloat16, {}),
    (5, 203, 192, 64, torch.float32, {}),
    (13, 390, 192, 64, torch.float32, dict(causal=0)),
])
def test_a_replayed_relay_equals_an_eager_one(P, n_q, n_k, d, dtype, extra):
    g = torch.Generator(device="cuda").manual_seed(n_q)
    cfg = dict(batch=1, heads=P, n_q=n_q, n_k=n_k, d=d, k=12, m=6, r=6, causal=1, causal_offset=max(0, n_k - n_q), seed=4,
               dtype=B.RR_BF16 if dtype == torch.bfloat16 else B.RR_F32)
    cfg.update(extra)
    rnd = lambda n: torch.randn((P, n, d), generator=g, device="cuda") * d ** -0.5
    q, k = rnd(n_q), rnd(n_k)
    data = []
    for _ in range(6):
        data.append((q.to(dtype), k.to(dtype)))
        q, k = (0.995 * x + 0.1 * rnd(x.shape[1]) for x in (q, k))
    led, ref = (RouteLedger(B.rr_config(**cfg)) for _ in range(2))
    buf = tuple(x.clone() for x in data[0])
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    for x in (led, ref):
        x.route_anchor(*data[0], 0)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
        led.route_relay(*buf, 1)
    flagged = 0
    for l in range(1, 6):
        for b, x in zip(buf, data[l]):
            b.copy_(x)
        torch.cuda.synchronize()
        if l < 5:
            graph.replay()
        else:
            led.route_relay(*buf, 1)                 # an eager call behind an odd number of recorded ones
        torch.cuda.synchronize()
        ref.route_relay(*data[l], 1)
        assert led.status() == 0 and ref.status() == 0
        n = int(led.refresh_count.item())
        want = torch.nonzero(led.flags).flatten().int()
        assert n == want.numel() and torch.equal(led.refresh_rows[:n], want), l
        counts = led.flags.view(P, n_q).sum(dim=1, dtype=torch.int32)
        assert torch.equal(led.problem_offsets[1:], counts.cumsum(0, dtype=torch.int32)), l
        for f in FIELDS:
            assert torch.equal(getattr(led, f), getattr(ref, f)), (f, l)
        flagged += n
    assert flagged > 0
    del graph
    led.close(); ref.close()
