"""The threshold form of the greedy step against the oracle, bit for bit, on
both sides of 256 experts: a warp's sorted lists up to there, the block's sort
(block_sort.cuh) beyond, around the sizes it rounds to; no, some and all of the
mass covered, ties, warm-up sets and sparse scores."""
import pytest

from paper_2602_07265_gb300 import workloads as W
from test_gpu_route import X, check  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 5, 31, 32, 33, 64, 65, 256, 257, 511, 512, 513, 800, 1000, 1024])
@pytest.mark.parametrize("tau", [0.0, 0.4, 0.9, 1.0])
@pytest.mark.parametrize("B,k0,sparse,ties", [(20, 1, 0, False), (70, 0, 0, True), (40, 0, 1, False)])
def test_threshold(X, N, tau, B, k0, sparse, ties):  # noqa: F811
    p = W.random_scores(B, N, seed=N + B, ties=ties)
    check(X, p, min(8, N), 0, W.MODE_THRESH, k0=k0, tau=tau, sparse_scores=sparse)
