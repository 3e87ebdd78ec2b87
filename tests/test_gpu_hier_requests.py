"""Algorithm 3 for request lengths that do not divide a 32-token chunk (the
chunk a request begins in selects it, with its tokens of the next chunk), at
the lengths around the limit and where the scores no longer fit on one SM:
against the oracle, bit for bit."""
import pytest

from paper_2602_07265_gb300 import workloads as W
from test_gpu_route import X, check  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,R,N", [
    (3, 10, 64), (5, 25, 128), (5, 13, 64), (7, 10, 200), (12, 30, 256), (31, 5, 256), (32, 3, 100),
    (33, 4, 64), (6, 40, 1000), (18, 6, 1000), (17, 6, 1024), (5, 400, 96)])
@pytest.mark.parametrize("sparse", [0, 1])
def test_request_lengths(X, T, R, N, sparse):  # noqa: F811
    for k0, m_r, budget, ties in ((1, 4, 0, False), (0, 3, 8, True), (2, 1, 5, False)):
        p = W.random_scores(T * R, N, seed=T + N, ties=ties)
        check(X, p, 8, budget, W.MODE_HIER, k0=k0, m_r=m_r, tokens_per_request=T, sparse_scores=sparse)
