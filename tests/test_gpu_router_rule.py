"""The routers on both sides of the line between CUDA cores and tensor cores:
the scores against 64 bits, and the forward against the oracle."""
import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_forward import P_RTOL, compare, gpu_forward
from test_gpu_route import X  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,d,B", [
    (64, 2048, 63), (64, 2048, 64), (64, 2048, 256), (64, 2048, 257), (100, 512, 655), (100, 512, 656),
    (8, 3968, 1057), (8, 3968, 1058), (9, 4096, 64), (1024, 128, 256), (1024, 128, 257),
    (128, 128, 192), (128, 128, 193), (32, 256, 768), (32, 256, 769), (16, 2048, 1024), (16, 2048, 1025),
    (66, 512, 3000), (130, 512, 8191), (132, 512, 8191)])
def test_both_routers(X, N, d, B):  # noqa: F811
    w = W.TINY.with_(N=N, d=d, F=128, B=B, k=4, budget=6)
    x, W_g = W.router_inputs(w, seed=9)
    weights = W.expert_weights(w, seed=9, device="cuda")
    g = gpu_forward(X, w, x, W_g, weights)
    p = torch.softmax(x.double() @ W_g.double().T, dim=1)
    assert ((torch.from_numpy(g["p"]).double() - p).abs() / p).max() <= P_RTOL
    compare(w, g, x, W_g, weights)
