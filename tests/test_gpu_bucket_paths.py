"""The buckets of a set run side by side: whether a relay's test runs inside the routing kernel goes by the row tiles of the
whole set (up to half of the SMs), and either way a bucket's results are those of a ledger of its own."""
import pytest
import torch

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200.ledger import BucketSet, RouteLedger

pytestmark = pytest.mark.gpu

WIDTHS = (8, 16, 32)
FIELDS = ("routes", "sentinels", "ages", "kth_score", "margin", "flags", "problem_offsets", "refresh_count")


@pytest.mark.parametrize("tiles", ["few", "half", "above_half", "many"])
def test_buckets_count_their_tiles_together(tiles):
    half = torch.cuda.get_device_properties(0).multi_processor_count // 2
    P = {"few": 3, "half": half // 3 * 3, "above_half": half // 3 * 3 + 3, "many": 2 * half + 3}[tiles]
    n_q, n_k, d = 100, 200, 64                               # (one row tile per problem)
    g = torch.Generator(device="cuda").manual_seed(P)
    rnd = lambda n: torch.randn((P, n, d), generator=g, device="cuda") * d ** -0.5
    cfg = dict(batch=1, n_q=n_q, n_k=n_k, d=d, m=8, r=8, dtype=B.RR_BF16, causal=1, causal_offset=100, seed=2)
    bs = BucketSet(B.rr_config(heads=P, k=1, **cfg), [WIDTHS[p % 3] for p in range(P)])
    alone = [RouteLedger(B.rr_config(heads=inf.problems, k=inf.k, **cfg)) for inf in bs.info]
    q, k = rnd(n_q), rnd(n_k)
    for l in range(4):
        qb, kb = q.bfloat16(), k.bfloat16()
        torch.cuda.synchronize()
        before = B.rr_kernel_launch_count()
        bs.route_layer(qb, kb, l, l == 0)
        launched = B.rr_kernel_launch_count() - before
        torch.cuda.synchronize()
        for inf, led, ref in zip(bs.info, bs.buckets, alone):
            part = slice(inf.first_slot, inf.first_slot + inf.problems)
            (ref.route_anchor if l == 0 else ref.route_relay)(qb[part], kb[part], l)
            for f in FIELDS:
                assert torch.equal(getattr(led, f), getattr(ref, f)), (inf.k, f, l)
        if l > 0:
            assert launched == 3 * (2 if tiles in ("few", "half") else 3)
        q, k = (0.99 * x + 0.14 * rnd(x.shape[1]) for x in (q, k))
    assert bs.status() == 0 and all(x.status() == 0 for x in alone)
    bs.close()
    for x in alone:
        x.close()
