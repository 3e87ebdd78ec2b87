"""The permutation of batches of more than two 32-token chunks (the chunks'
counts are combined by one CTA, the pairs placed by the next kernel): sizes at
the edges of its chunks, experts and parts, against the oracle bit for bit,
and the same rows through the layer forward's gather."""
import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_forward import compare, gpu_forward
from test_gpu_route import X, check  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,k", [
    (65, 1, 1), (65, 33, 16), (96, 31, 3), (97, 64, 8), (129, 257, 8), (160, 512, 5),
    (1000, 48, 7), (1024, 1024, 16), (2049, 96, 8), (8192, 64, 8), (8161, 300, 2)])
def test_route_permutation_sizes(X, B, N, k):  # noqa: F811
    p = W.random_scores(B, N, seed=B + N, ties=B % 2 == 0)
    check(X, p, k, min(N, 24), W.MODE_BATCH, k0=1 if N > 1 else 0)
    check(X, p, k, 0, W.MODE_TOPK)


@pytest.mark.parametrize("B,n_shared", [(65, 0), (200, 2), (1300, 1)])
def test_forward_gathers_the_permuted_rows(X, B, n_shared):  # noqa: F811
    w = W.TINY.with_(B=B, d=256, F=128, budget=20)
    x, W_g = W.router_inputs(w, seed=3)
    weights = W.expert_weights(w, seed=3, device="cuda")
    shared = W.shared_expert_weights(w, n_shared, seed=3) if n_shared else None
    g = gpu_forward(X, w, x, W_g, weights, shared=shared)
    compare(w, g, x, W_g, weights, shared=shared)
    assert g["stats"]["status"] == 0 and torch.isfinite(torch.from_numpy(g["y"])).all()
