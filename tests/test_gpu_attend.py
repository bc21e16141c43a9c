"""The consumer of token ranges at its edges: head widths with and without 16-byte lanes, token
counts around the 32-token blocks and the four warps' share, empty rows and slots, ranges past the
last token."""
import pytest
import torch

from paper_2609_07306_b200.ledger import attend_token_ranges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dh", [(torch.bfloat16, 64), (torch.bfloat16, 128), (torch.bfloat16, 256),
                                      (torch.float32, 32), (torch.float32, 64), (torch.float32, 128),
                                      (torch.bfloat16, 40), (torch.float32, 20)])
def test_token_counts_and_head_widths(dtype, dh):
    g = torch.Generator(device="cuda").manual_seed(dh)
    P, n_q, tokens, slots = 2, 12, 700, 5
    spans = [[], [(3, 4)], [(0, 31)], [(0, 32)], [(5, 38)], [(0, 127), (200, 201)], [(1, 129)], [(0, 128), (128, 256)],
             [(10, 20), (30, 300), (699, 700)], [(650, 900)], [(0, 700)], [(0, 1), (2, 3), (4, 5), (6, 7), (698, 705)]]
    rg = torch.full((P * n_q, slots, 2), -1, dtype=torch.int32)
    for p in range(P):
        for i, sp in enumerate(spans):
            for s, (lo, hi) in enumerate(sp):
                slot = s if p == 0 else slots - len(sp) + s            # empty slots in front, too
                rg[p * n_q + i, slot] = torch.tensor([lo, hi])
    q, k, v = (torch.randn(shape, generator=g, device="cuda").to(dtype)
               for shape in ((P * n_q, dh), (P, tokens, dh), (P, tokens, dh)))
    out = attend_token_ranges(rg.cuda(), n_q, q, k, v, dh ** -0.5)
    for r in range(P * n_q):
        p, sp = r // n_q, spans[r % n_q]
        if not sp:
            assert (out[r] == 0).all()
            continue
        idx = torch.cat([torch.arange(lo, min(hi, tokens)) for lo, hi in sp]).cuda()
        kk, vv = k[p, idx].double(), v[p, idx].double()
        want = torch.softmax(kk @ q[r].double() * dh ** -0.5, 0) @ vv
        torch.testing.assert_close(out[r].double(), want, rtol=2e-5, atol=2e-6)
