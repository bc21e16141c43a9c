"""The consumer of token ranges at its edges: head widths with and without 16-byte lanes, token
counts around the 32-token blocks and the four warps' share, empty rows and slots, ranges past the
last token, tokens masked by their logits, infinities beside the last token."""
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


@pytest.mark.parametrize("dtype,dh", [(torch.bfloat16, 128), (torch.float32, 64), (torch.float32, 20)])
@pytest.mark.parametrize("mask", [float("-inf"), "lowest"])
def test_tokens_masked_by_their_keys(dtype, dh, mask):
    """Keys that make a token's logit -inf (an infinity, or the type's lowest value, which overflows):
    such tokens weigh nothing, also where a whole block or a whole warp's share is masked; a row with
    nothing else has no softmax."""
    g = torch.Generator(device="cuda").manual_seed(dh)
    tokens, n_q = 330, 6
    low = torch.finfo(dtype).min if mask == "lowest" else mask
    q = (torch.rand((n_q, dh), generator=g, device="cuda") + 2.0).to(dtype)        # (lowest value times more than 1)
    k, v = (torch.randn((1, tokens, dh), generator=g, device="cuda").to(dtype) for _ in range(2))
    k[0, 0:40] = low                             # the first block, and more
    k[0, 96:128] = low                           # the first share of the fourth warp
    k[0, 200] = low
    spans = [(0, 330), (0, 128), (0, 45), (96, 130), (0, 32), (190, 210)]
    rg = torch.tensor(spans, dtype=torch.int32, device="cuda").view(n_q, 1, 2)
    out = attend_token_ranges(rg, n_q, q, k, v, dh ** -0.5)
    off = torch.zeros(tokens, dtype=torch.bool, device="cuda")
    for lo, hi in ((0, 40), (96, 128), (200, 201)):
        off[lo:hi] = True
    for i, (lo, hi) in enumerate(spans):
        idx = torch.arange(lo, hi, device="cuda")
        idx = idx[~off[idx]]
        if idx.numel() == 0:
            assert out[i].isnan().all()
            continue
        want = torch.softmax(k[0, idx].double() @ q[i].double() * dh ** -0.5, 0) @ v[0, idx].double()
        torch.testing.assert_close(out[i].double(), want, rtol=2e-5, atol=2e-6)


@pytest.mark.parametrize("dtype,dh", [(torch.bfloat16, 128), (torch.float32, 64), (torch.float32, 20)])
def test_infinite_value_at_the_last_token(dtype, dh):
    """An infinity in the last token's value row, where the last block of 32 is partly empty: inf, not NaN."""
    g = torch.Generator(device="cuda").manual_seed(dh)
    q = torch.randn((1, dh), generator=g, device="cuda").to(dtype)
    k, v = (torch.randn((1, 50, dh), generator=g, device="cuda").to(dtype) for _ in range(2))
    v[0, 39, 0] = float("inf")
    out = attend_token_ranges(torch.tensor([[[0, 40]]], dtype=torch.int32, device="cuda"), 1, q, k, v, dh ** -0.5)
    assert torch.isposinf(out[0, 0]) and torch.isfinite(out[0, 1:]).all()
