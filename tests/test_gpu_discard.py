"""The kernels that discard dead lines.  The combine (outputs, activations):
sizes on both sides of its line (6 MB of expert outputs), more rows a token than
a warp takes at once, rows of activations shorter and longer than the warps'
shares, shared experts.  The down kernels (gathered tokens, 16 to 64 MB): at both
ends, both kernels."""
import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_forward import compare, gpu_forward
from test_gpu_route import X  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,d,F,k,n_shared,mode", [
    (191, 1024, 128, 8, 0, W.MODE_BATCH),    # just below the line
    (192, 1024, 128, 8, 0, W.MODE_BATCH),    # on it; 2 activation lines for 8 warps of columns
    (600, 256, 1152, 9, 2, W.MODE_TOPK),     # 18 activation lines for 2 warps, 11 rows a token
    (130, 1152, 640, 16, 0, W.MODE_BATCH),   # 9 warps of columns, the second block partly empty
    (1024, 1024, 128, 8, 0, W.MODE_BATCH),   # 16 MB of tokens, CTA pairs
    (910, 1024, 128, 8, 1, W.MODE_TOPK),     # just below
    (150, 8192, 128, 7, 1, W.MODE_TOPK),     # 18.75 MB with few tokens an expert, shared rows
    (4096, 1024, 128, 8, 0, W.MODE_TOPK),    # 64 MB
    (4097, 1024, 128, 8, 0, W.MODE_TOPK),    # just above
])
def test_discard(X, B, d, F, k, n_shared, mode):  # noqa: F811
    w = W.TINY.with_(B=B, N=24 if d < 8192 else 120, d=d, F=F, k=k, budget=18, mode=mode)
    x, W_g = W.router_inputs(w, seed=4)
    weights = W.expert_weights(w, seed=4, device="cuda")
    shared = W.expert_weights(w.with_(N=n_shared), seed=5, device="cuda") if n_shared else None
    g = gpu_forward(X, w, x, W_g, weights, shared)
    compare(w, g, x, W_g, weights, shared=shared)

    # Calls in turn on one workspace, nothing between them: the same bits.
    prm = X.route_params(**w.params())
    ws = torch.empty(X.xshare_workspace_size(B, w.N, k, d, F, mode, prm, n_shared), dtype=torch.uint8,
                     device="cuda")
    xs = [x.cuda(), W.router_inputs(w, seed=6)[0].cuda()]
    W_g = W_g.cuda()
    ys = [torch.empty(B, d, dtype=torch.bfloat16, device="cuda") for _ in range(6)]
    for i, y in enumerate(ys):
        X.xshare_moe_forward(xs[i % 2], W_g, *weights, k, w.budget, mode, prm, y, ws, shared=shared)
    torch.cuda.synchronize()
    assert (ys[0].cpu().float().numpy() == g["y"]).all()
    for i in range(2, 6):
        assert torch.equal(ys[i], ys[i % 2])
