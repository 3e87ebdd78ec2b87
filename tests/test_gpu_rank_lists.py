"""Ranking with more than 256 experts (unsorted lane lists of 16 and 32) against
the oracle, bit for bit: ties, every mode, both sides of 512 experts, |S| on
both sides of each compact list length."""
import pytest

from paper_2602_07265_gb300 import workloads as W
from test_gpu_route import X, check  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,B,k,mode,budget,prm", [
    (257, 33, 16, W.MODE_TOPK, 0, {}), (512, 40, 16, W.MODE_TOPK, 0, {}), (513, 40, 16, W.MODE_TOPK, 0, {}),
    (512, 97, 8, W.MODE_BATCH, 257, dict(k0=1)), (384, 66, 8, W.MODE_HIER, 3, dict(k0=1, m_r=5, tokens_per_request=3)), (1024, 40, 16, W.MODE_TOPK, 0, {}),
    (512, 70, 8, W.MODE_BATCH, 64, dict(k0=0)), (512, 70, 8, W.MODE_BATCH, 65, dict(k0=0)),
    (700, 97, 8, W.MODE_BATCH, 128, dict(k0=0)), (700, 97, 8, W.MODE_BATCH, 256, dict(k0=0)),
    (1000, 97, 8, W.MODE_BATCH, 257, dict(k0=0)), (960, 66, 5, W.MODE_GROUP, 0, dict(k0=2, n_groups=4, m_g=40)),
    (333, 64, 8, W.MODE_HIER, 3, dict(k0=1, m_r=5, tokens_per_request=4)),
    (600, 32, 8, W.MODE_THRESH, 0, dict(k0=1, tau=0.6)),
    (400, 65, 4, W.MODE_BATCH, 30, dict(k0=3, sparse_scores=1))])
@pytest.mark.parametrize("ties", [False, True])
def test_long_lists(X, N, B, k, mode, budget, prm, ties):  # noqa: F811
    check(X, W.random_scores(B, N, seed=N, ties=ties), k, budget, mode, **prm)
