"""The CTA-pair FFN kernels (many tokens per expert) against the oracle, on
plain and packed weights (the same bits), at the edges of their tiles: token
counts around 32 and 256, an odd number of 128-row blocks in d, two K steps,
experts with few tokens beside full ones, shared experts, few tokens per
expert (batches of one, two and five 32-token chunks), repeated calls, and the
ranks of an expert-parallel layer."""
import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_ep import run_ep, run_one_gpu
from test_gpu_forward import compare, gpu_forward
from test_gpu_route import X  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _inputs(w, n_shared):
    x, W_g = W.router_inputs(w, seed=5)
    weights = W.expert_weights(w, seed=5, device="cuda")
    return x, W_g, weights, W.shared_expert_weights(w, n_shared, seed=5) if n_shared else None


# With N == k every expert gets exactly B tokens; otherwise the counts spread.
@pytest.mark.parametrize("N,k,d,F,B,mode,n_shared", [
    (2, 2, 128, 128, 64, W.MODE_TOPK, 0), (4, 4, 384, 256, 255, W.MODE_TOPK, 0),
    (2, 2, 256, 384, 256, W.MODE_TOPK, 1), (3, 3, 640, 128, 257, W.MODE_TOPK, 0),
    (8, 2, 256, 256, 1000, W.MODE_TOPK, 2), (32, 4, 128, 384, 700, W.MODE_BATCH, 0),
    (16, 3, 2048, 256, 513, W.MODE_HIER, 0), (2, 2, 512, 128, 30, W.MODE_TOPK, 0),
    (38, 8, 512, 256, 63, W.MODE_TOPK, 1), (38, 4, 512, 256, 150, W.MODE_TOPK, 0),
    # few experts, long units (112 steps on 8 of the pairs; two rounds of 112), and the other side of the rule
    (4, 2, 7168, 256, 64, W.MODE_TOPK, 0), (4, 2, 7168, 2560, 100, W.MODE_TOPK, 0),
    (4, 2, 7168, 256, 48, W.MODE_TOPK, 0)])
def test_pair_forward(X, N, k, d, F, B, mode, n_shared):  # noqa: F811
    w = W.TINY.with_(N=N, k=k, d=d, F=F, B=B, mode=mode, budget=6, k0=0, m_r=2,
                     tokens_per_request=3 if mode == W.MODE_HIER else 1, x_kind="domains")
    x, W_g, weights, shared = _inputs(w, n_shared)
    g = gpu_forward(X, w, x, W_g, weights, shared=shared)
    assert g["stats"]["status"] == 0
    compare(w, g, x, W_g, weights, shared=shared)
    pk, ps = X.Packed(*weights), X.Packed(*shared) if shared else None
    y = run_one_gpu(X, w, x, W_g, pk, shared=ps)["y"]
    assert torch.equal(y, run_one_gpu(X, w, x, W_g, pk, shared=ps)["y"])
    assert torch.equal(y.cpu().double(), torch.from_numpy(g["y"])), "packed and plain weights differ"


def test_pair_rounds_like_the_other_path(X):  # noqa: F811
    """A token's output does not depend on the path: 8 experts of 18 blocks are
    whole units on either (ffn_tc.cu gives each of 144 CTAs one), so that a
    batch of 7 tokens, which ffn_tc.cu takes, has the bits of the same tokens
    in a batch of 256, which the pairs take."""
    w = W.TINY.with_(N=8, k=8, d=2304, F=2304, B=256, mode=W.MODE_TOPK, budget=0, k0=0)
    x, W_g, weights, _ = _inputs(w, 0)
    pk = X.Packed(*weights)
    y = run_one_gpu(X, w, x, W_g, pk)["y"]
    for t in range(0, w.B - 7, 7):
        few = run_one_gpu(X, w.with_(B=7), x[t:t + 7].contiguous(), W_g, pk)["y"]
        assert torch.equal(few, y[t:t + 7])


def test_pair_expert_parallel(X):  # noqa: F811
    w = W.TINY.with_(N=8, k=2, d=256, F=256, B=900, mode=W.MODE_TOPK, x_kind="domains")
    x, W_g, weights, shared = _inputs(w, 1)
    pk, ps = X.Packed(*weights), X.Packed(*shared)
    one = run_one_gpu(X, w, x, W_g, pk, shared=ps)["y"]
    y = run_ep(X, w, x, W_g, pk, 4, shared=ps)[0]
    assert torch.equal(y, one)   # no unit is cut: every row is the same bits on any rank


def test_pair_graph_and_streams(X):  # noqa: F811
    """A stack captured into a graph gives the direct call's bits; forwards on
    two streams with workspaces of their own give the results they give alone."""
    w = W.TINY.with_(N=8, k=2, d=256, F=256, B=600, mode=W.MODE_TOPK, x_kind="domains")
    x, W_g, weights, _ = _inputs(w, 0)
    dev = torch.device("cuda")
    prm, pk, x, W_g = X.route_params(**w.params()), X.Packed(*weights), x.to(dev), W_g.to(dev)
    size = X.xshare_workspace_size(w.B, w.N, w.k, w.d, w.F, w.mode, prm)
    ws = [torch.empty(size, dtype=torch.uint8, device=dev) for _ in range(3)]
    layers = [(W_g, pk)] * 3
    h = [torch.empty(3, w.B, w.d, dtype=torch.bfloat16, device=dev) for _ in range(2)]
    X.xshare_stack_forward(x, layers, w.k, 0, w.mode, prm, h[0], ws[0])
    torch.cuda.synchronize()
    g = X.StackGraph(x, layers, w.k, 0, w.mode, prm, h[1], ws[1])
    for _ in range(3):
        g.launch()
    torch.cuda.synchronize()
    assert torch.equal(h[0].view(torch.int16), h[1].view(torch.int16))
    xs = [x, x.flip(0).contiguous()]
    alone = [torch.empty_like(x) for _ in xs]
    both = [torch.empty_like(x) for _ in xs]
    for i, xi in enumerate(xs):
        X.xshare_moe_forward_packed(xi, W_g, pk, w.k, 0, w.mode, prm, alone[i], ws[0])
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    for _ in range(5):
        for i, xi in enumerate(xs):
            X.xshare_moe_forward_packed(xi, W_g, pk, w.k, 0, w.mode, prm, both[i], ws[1 + i], stream=streams[i])
    torch.cuda.synchronize()
    for a, b in zip(alone, both):
        assert torch.equal(a.view(torch.int16), b.view(torch.int16))
