"""Batches around the line below which the gather kernel warms nothing (more
selected experts than pairs): packed and plain weights give the same bits and
match the oracle on both sides of it."""
import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_ep import run_one_gpu
from test_gpu_forward import compare, gpu_forward
from test_gpu_route import X  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,budget", [(1, 7), (1, 8), (1, 9), (2, 16), (2, 17), (3, 24), (3, 25)])
def test_few_pairs(X, B, budget):  # noqa: F811
    w = W.TINY.with_(B=B, budget=budget)
    x, W_g = W.router_inputs(w, seed=6)
    weights = W.expert_weights(w, seed=6, device="cuda")
    g = gpu_forward(X, w, x, W_g, weights)
    compare(w, g, x, W_g, weights)
    y = run_one_gpu(X, w, x, W_g, X.Packed(*weights))["y"]
    assert torch.equal(y.cpu().double(), torch.from_numpy(g["y"]))
