"""Plain top-k in one kernel (more than two 32-token chunks) against the oracle,
bit for bit (route), and through the forward."""
import pytest

from paper_2602_07265_gb300 import workloads as W
from test_gpu_forward import compare, gpu_forward
from test_gpu_route import X, check  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,k", [(65, 8, 8), (96, 64, 1), (1000, 128, 8), (2500, 200, 16), (100, 700, 5)])
def test_topk(X, B, N, k):  # noqa: F811
    check(X, W.random_scores(B, N, seed=B, ties=N == 128), k, 0, W.MODE_TOPK, n_groups=2 if N % 2 == 0 else 1)


@pytest.mark.parametrize("B", [70, 300])
def test_topk_forward(X, B):  # noqa: F811
    w = W.TINY.with_(B=B, mode=W.MODE_TOPK)
    x, W_g = W.router_inputs(w, seed=8)
    weights = W.expert_weights(w, seed=8, device="cuda")
    compare(w, gpu_forward(X, w, x, W_g, weights), x, W_g, weights)
