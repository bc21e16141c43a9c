"""Small grids test a relay's rows inside the routing kernel, larger ones in a kernel of their own with a list between.
The rows of a ledger's first problems do not depend on how many problems follow (rows are numbered problem by
problem), so both ways can be held against each other bit for bit."""
import pytest
import torch

from paper_2609_07306_b200 import binding as B
from paper_2609_07306_b200.ledger import RouteLedger

pytestmark = pytest.mark.gpu

LAYERS = 4
FIELDS = ("routes", "sentinels", "ages", "kth_score", "margin", "flags", "alpha", "beta")


def _inputs(P, n_q, n_k, d, rho, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    def rnd(n): return torch.randn((P, n, d), generator=g, device="cuda") * d ** -0.5
    mu = rnd(16)
    pick = lambda n: mu.gather(1, torch.randint(0, 16, (P, n), generator=g, device="cuda")[:, :, None].expand(P, n, d))
    q, k = pick(n_q) + 0.5 * rnd(n_q), pick(n_k) + 0.5 * rnd(n_k)
    out = []
    for _ in range(LAYERS):
        out.append((q.bfloat16(), k.bfloat16()))
        q, k = ((1 - rho * rho) ** 0.5 * x + rho * rnd(x.shape[1]) for x in (q, k))
    return out


# (widths at every column capacity; no sentinels, global sentinels, ragged tiles, chunks around the 64 of a tile,
# rows that see fewer chunks than they keep, policies, ranges; one row, no drift, strong drift)
@pytest.mark.parametrize("n_q,n_k,d,k,m,r,rho,extra", [
    (256, 256, 128, 16, 8, 8, 0.15, {}),
    (129, 193, 64, 24, 4, 5, 0.05, dict(global_sentinels=3)),
    (150, 700, 128, 28, 8, 0, 0.02, dict(causal_offset=550)),
    (100, 63, 64, 32, 8, 9, 0.3, {}),
    (300, 1024, 128, 32, 16, 16, 0.1, dict(gamma=0.01, min_reuse=1, h_max=2)),
    (128, 65, 128, 40, 16, 3, 0.1, dict(causal=0)),
    (260, 512, 64, 50, 18, 12, 0.01, dict(chunk_tokens=16)),
    (128, 512, 64, 40, 28, 16, 0.2, {}),
    (130, 320, 128, 50, 30, 32, 0.1, dict(gamma_boost=0.05, margin_recover=0.01)),
    (140, 2048, 128, 64, 32, 32, 0.15, {}),
    (1, 1100, 64, 20, 0, 0, 0.1, dict(causal=0)),
    (200, 400, 128, 12, 12, 12, 0.0, {}),
])
@pytest.mark.parametrize("slow_rows", [0, 8])
def test_small_grid_equals_the_first_problems_of_a_large_one(n_q, n_k, d, k, m, r, rho, extra, slow_rows):
    few = 2
    tiles = (n_q + 127) // 128
    many = torch.cuda.get_device_properties(0).multi_processor_count // tiles + 1
    data = _inputs(many, n_q, n_k, d, rho, seed=n_q + n_k)
    cfg = dict(batch=1, n_q=n_q, n_k=n_k, d=d, k=k, m=m, r=r, dtype=B.RR_BF16, causal=1, causal_offset=0, seed=3,
               debug_outputs=slow_rows)
    cfg.update(extra)
    small, large = (RouteLedger(B.rr_config(heads=P, **cfg)) for P in (few, many))
    launched = []
    for l, (q, kk) in enumerate(data):
        for led, P in ((small, few), (large, many)):
            before = B.rr_kernel_launch_count()
            (led.route_anchor if l == 0 else led.route_relay)(q[:P].contiguous(), kk[:P].contiguous(), l)
            launched.append(B.rr_kernel_launch_count() - before)
        assert small.status() == 0 and large.status() == 0
        rows = few * n_q
        for f in FIELDS + (("token_ranges",) if cfg.get("chunk_tokens") else ()):
            a, b = getattr(small, f), getattr(large, f)[:rows]
            assert torch.equal(a.view(torch.int32) if a.dtype == torch.float32 else a,
                               b.view(torch.int32) if b.dtype == torch.float32 else b), (f, l)
        n = int(small.refresh_count.item())
        assert torch.equal(small.refresh_rows[:n], torch.nonzero(small.flags).flatten().int())
        assert torch.equal(small.problem_offsets, large.problem_offsets[:few + 1])
    assert launched[2] == launched[3] - 1                    # (the test has no launch of its own)
    for led in (small, large):
        led.close()
