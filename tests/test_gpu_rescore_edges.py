"""The challenge test's kernel where its reading of the ledger rows can go wrong: rows that do not split
into 16-byte loads, no sentinels at all, more loads than one batch, row tiles and quarters that end
early, key chunks that end inside a bitmap word."""
import pytest

import parity
from paper_2609_07306_b200 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_q,n_k,d,k,m,r,causal", [
    (1, 40, 64, 1, 0, 1, False), (31, 65, 128, 4, 4, 4, True), (33, 97, 64, 5, 3, 0, True),
    (97, 300, 128, 3, 0, 0, False), (129, 333, 64, 64, 32, 31, False), (160, 2048, 128, 9, 1, 8, True),
])
def test_ledger_rows_of_all_widths(n_q, n_k, d, k, m, r, causal):
    w = W.RouteWorkload("edge", 1, 3, n_q, n_k, d, k, m, r, layers=4, anchor_every=100, dtype=W.DTYPE_BF16,
                        centroids=10, rho=0.2, causal=causal, causal_offset=max(0, n_k - n_q), seed=8)
    parity.assert_clean(parity.run_teacher_forced(w))
