"""Host threads that call the library at the same time, each with a workspace
and a stream of its own, over calls whose kernels take different amounts of
shared memory: every call must be launched and give what it gives alone."""
import threading

import pytest
import torch

from paper_2602_07265_gb300 import workloads as W
from test_gpu_graph_streams import X, setup  # noqa: F401  (X: fixture)

pytestmark = pytest.mark.gpu


def run_threads(makers, n_calls):
    """makers: functions that return (call, result).  Each call runs alone
    first; then all of them n_calls times at once, a thread each."""
    calls, alone, errors = [], [], []
    for make in makers:
        call, result = make()
        call(None)
        torch.cuda.synchronize()
        alone.append([t.clone() for t in result])
        calls.append((call, result))
    start = threading.Barrier(len(calls))

    def work(call):
        s = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(n_calls):
                call(s)
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        s.synchronize()

    threads = [threading.Thread(target=work, args=(c,)) for c, _ in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for (_, result), want in zip(calls, alone):
        for got, w in zip(result, want):
            assert torch.equal(got, w)


@pytest.mark.parametrize("N", [512, 1024])
def test_selection_kernel(X, N):  # noqa: F811
    """score_kernel of one expert count: HIER requests across chunk edges take
    more rows than BATCH."""
    def maker(mode, **kw):
        def make():
            B, k = 40, 8
            p = torch.from_numpy(W.random_scores(B, N, seed=N + mode)).cuda()
            prm = X.route_params(k0=1, **kw)
            ws = torch.empty(X.xshare_workspace_size(B, N, k, 0, 0, mode, prm), dtype=torch.uint8, device="cuda")
            mask = torch.empty(N, dtype=torch.uint8, device="cuda")
            ids = torch.empty(B, k, dtype=torch.int32, device="cuda")
            w = torch.empty(B, k, dtype=torch.float32, device="cuda")
            return (lambda s: X.xshare_route(p, k, 16, mode, prm, mask, ids, w, ws, stream=s)), (mask, ids, w)
        return make
    run_threads(2 * [maker(W.MODE_HIER, m_r=2, tokens_per_request=5), maker(W.MODE_BATCH)], 20000)


def test_sliced_router(X):  # noqa: F811
    """router_split_kernel of one batch class: wider layers take longer slices."""
    def maker(d):
        def make():
            w = W.TINY.with_(N=16, k=4, d=d, F=128, B=20, budget=4)
            pk, W_g, prm, ws = setup(X, w, 1)
            x = W.router_inputs(w, 2)[0].cuda()
            y = torch.empty(w.B, d, dtype=torch.bfloat16, device="cuda")
            return (lambda s: X.xshare_moe_forward_packed(x, W_g, pk, w.k, w.budget, w.mode, prm, y, ws,
                                                          stream=s)), (y,)
        return make
    run_threads(2 * [maker(4096), maker(16384)], 1500)
