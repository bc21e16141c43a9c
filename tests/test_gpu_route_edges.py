"""The two-threads-per-row routing kernel at the edges of its dispatch and of its tiles: column
capacities (keep = k + max(m, 1) at 28 | 29, 36 | 37, 48 | 49, 96 | 97, and by the number of key chunks), key chunks
around the 64-wide tiles and the two-tile round of a row's threads, rows that see fewer chunks than
they keep, ragged row tiles and widths that rule out 16-byte stores."""
import random

import numpy as np
import pytest
import torch

import parity
from paper_2609_07306_b200 import workload as W
from paper_2609_07306_b200.ledger import RouteLedger, config_from_workload, device_tensor

pytestmark = pytest.mark.gpu


def _w(n_q, n_k, d, k, m, r, causal, **kw):
    return W.RouteWorkload("edge", 1, 2, n_q, n_k, d, k, m, r, layers=3, anchor_every=100, dtype=W.DTYPE_BF16,
                           centroids=12, rho=0.2, causal=causal, seed=21, **kw)


@pytest.mark.parametrize("k,m", [(20, 8), (20, 9), (24, 12), (24, 13), (32, 16), (33, 16), (47, 0), (16, 32), (32, 32), (33, 32), (48, 32), (49, 32), (64, 32), (65, 32), (3, 1)])
def test_widths_around_the_column_capacities(k, m):
    rep = parity.run_teacher_forced(_w(150, 700, 128, k, m, 9, True, causal_offset=550))
    parity.assert_clean(rep)


@pytest.mark.parametrize("n_k", [1, 33, 63, 64, 65, 127, 128, 129, 192, 193, 1025])
def test_key_chunks_around_the_tiles(n_k):
    k = min(12, n_k)
    rep = parity.run_teacher_forced(_w(129, n_k, 64, k, min(8, n_k - k), 5, False))
    parity.assert_clean(rep)
    rep = parity.run_teacher_forced(_w(131, n_k, 128, k, 8, 5, True))
    parity.assert_clean(rep)


def test_best_chunks_in_one_threads_tiles():
    """Scores whose best chunks all lie in even tiles (one thread's share of every row), then in a
    handful of columns: the bound follows, routes stay exact."""
    w = _w(128, 1024, 64, 32, 16, 16, False)
    rng = np.random.default_rng(5)
    q = rng.standard_normal((2, 128, 64)).astype(np.float32)
    for boost in (lambda c: (c // 64) % 2 == 0, lambda c: c >= 1024 - 60, lambda c: c % 64 < 4):
        k = rng.standard_normal((2, 1024, 64)).astype(np.float32)
        k += np.where(boost(np.arange(1024)), 4.0, 0.0)[None, :, None] * q.mean(axis=1, keepdims=True)
        qb, kb = (W.f32_to_bf16_bits(x) for x in (q, k))
        led = RouteLedger(config_from_workload(w))
        led.route_anchor(device_tensor(qb), device_tensor(kb), 0)
        torch.cuda.synchronize()
        assert led.status() == 0
        s = np.einsum("pid,pjd->pij", W.bf16_bits_to_f32(qb).astype(np.float64), W.bf16_bits_to_f32(kb).astype(np.float64))
        want = np.sort(np.argsort(-s, axis=2)[:, :, :32], axis=2).reshape(-1, 32)
        got = led.routes.cpu().numpy()
        assert (got == want).all(axis=1).mean() > 0.999      # (float64 against fp32: near-ties only)
        led.close()


@pytest.mark.parametrize("n_q", [1, 32, 33, 65, 97, 128, 129])
@pytest.mark.parametrize("rho", [0.002, 0.2])
def test_quarters_without_rows(n_q, rho):
    """Row tiles whose last quarters (32 rows) are empty, at anchors and on short and long lists."""
    w = _w(n_q, 300, 64, 12, 8, 6, False).replace(rho=rho)
    parity.assert_clean(parity.run_teacher_forced(w))


# most kept chunks of the two-CTA columns and of the columns after them, by key chunks and head width, and
# the first that needs the next column
@pytest.mark.parametrize("n_k,d,keep", [
    (256, 128, 70), (256, 128, 71), (257, 128, 67), (320, 128, 66), (512, 128, 62), (513, 128, 62), (1024, 128, 58),
    (1025, 128, 57), (2048, 128, 56), (2049, 128, 56), (190, 128, 70), (256, 64, 76), (256, 64, 77), (320, 64, 72),
    (512, 64, 68), (1024, 64, 64), (1536, 64, 62), (1537, 64, 60), (256, 128, 92), (256, 64, 93), (320, 64, 80), (512, 128, 77), (1024, 64, 85)])
@pytest.mark.parametrize("causal", [False, True])
def test_columns_by_key_chunks(n_k, d, keep, causal):
    w = _w(131, n_k, d, keep - 24, 24, 9, causal, causal_offset=max(0, n_k - 131) if causal else 0)
    parity.assert_clean(parity.run_teacher_forced(w))


@pytest.mark.parametrize("n_k,keep", [(256, 71), (256, 76), (256, 77), (320, 72), (512, 68), (1024, 64), (1536, 62)])
def test_columns_of_grids_beyond_the_sms(n_k, keep):
    """The column that needs more CTAs than SMs to pay (d = 64): 160 problems, three of them checked."""
    w = _w(70, n_k, 64, keep - 20, 20, 7, True, causal_offset=n_k - 70).replace(heads=160, layers=2)
    parity.assert_clean(parity.run_teacher_forced(w, check_problems=[0, 77, 159]))


@pytest.mark.parametrize("k,m", [(64, 1), (65, 1), (1, 64), (1, 65), (45, 9)])
def test_wide_routes_of_unequal_parts(k, m):
    """Ids ordered per thread: up to 64 where two CTAs share an SM, more beyond."""
    parity.assert_clean(parity.run_teacher_forced(_w(140, 250, 64, k, m, 4, False)))


@pytest.mark.parametrize("n_k,d", [(256, 128), (200, 64)])
def test_slow_path_of_wide_routes(n_k, d):
    """Every fifth row through the exact slow path, then rows whose scores all tie (every row)."""
    w = _w(140, n_k, d, 40, 16, 8, True)
    parity.assert_clean(parity.run_teacher_forced(w, force_slow_rows=True))
    led = RouteLedger(config_from_workload(w))
    led.route_anchor(torch.zeros(2, 140, d, device="cuda", dtype=torch.bfloat16),
                     torch.zeros(2, n_k, d, device="cuda", dtype=torch.bfloat16), 0)
    torch.cuda.synchronize()
    r = led.routes.cpu().numpy().reshape(2, 140, 40)
    s = led.sentinels.cpu().numpy().reshape(2, 140, -1)[:, :, :16]
    for i in range(140):
        kk, nn = min(40, i + 1), min(16, max(0, i + 1 - 40))
        assert (np.sort(r[:, i, :kk], 1) == np.arange(kk)).all() and (r[:, i, kk:] == -1).all(), i
        assert (np.sort(s[:, i, :nn], 1) == np.arange(kk, kk + nn)).all() and (s[:, i, nn:] == -1).all(), i
    led.close()


@pytest.mark.parametrize("kind", ["normal", "ties", "one_threads_tiles", "duplicates", "large", "uneven"])
def test_wide_columns_equal_the_two_pass_path(kind):
    """Bit for bit, over random shapes of 49 to 96 kept chunks and scores that strain the bound: the exact
    select of the two-pass path runs on the same scores (same tile MMAs)."""
    rng = random.Random(kind)
    g = torch.Generator(device="cuda").manual_seed(3)
    for _ in range(8):
        d, n_q = rng.choice([64, 128]), rng.choice([1, 40, 131, 300])
        n_k = rng.choice([rng.randint(100, 330), rng.randint(100, 2100)])
        P = 170 if n_q == 40 and n_k < 600 else 2                          # (more CTAs than SMs)
        keep = rng.randint(49, 96)
        m = rng.choice([0, 1, 20, keep // 2, keep - 1])
        causal = rng.random() < 0.5
        w = _w(n_q, n_k, d, keep - max(m, 1), m, rng.choice([0, 5, 8]), causal, causal_offset=n_k // 2 if causal else 0,
               global_sentinels=rng.choice([0, 3])).replace(heads=P)
        q, k = (torch.randn((P, n, d), generator=g, device="cuda") for n in (n_q, n_k))
        if kind == "ties":
            q.round_(); k.round_()
        elif kind == "one_threads_tiles":
            k[:, (torch.arange(n_k, device="cuda") // 64) % 2 == 0] += 0.8 * q.mean((0, 1))
        elif kind == "duplicates":
            k = k[:, torch.randint(0, n_k // 3, (n_k,), generator=g, device="cuda")]
        elif kind == "large":
            q *= 1e18; k *= 1e18
        elif kind == "uneven":
            k *= torch.rand((P, n_k, 1), generator=g, device="cuda") ** 4
        q, k = q.bfloat16().contiguous(), k.bfloat16().contiguous()
        got = []
        for two_pass in (False, True):
            led = RouteLedger(config_from_workload(w, two_pass=two_pass))
            led.route_anchor(q, k, 3)
            led.route_relay(q, k, 4)
            assert led.status() == 0
            got.append([led.routes.sort(1).values, led.sentinels[:, :m].sort(1).values, led.sentinels[:, m:].clone(),
                        led.kth_score.clone(), led.margin.clone()])
            led.close()
        assert all(torch.equal(a, b) for a, b in zip(*got)), (w, [torch.equal(a, b) for a, b in zip(*got)])
