"""The rule that sends a batch to the CTA-pair FFN kernels (pair_rule.cuh), on
the CPU: the side that measured faster on GB300 (76 pairs at once) at layers
of few experts, of narrow experts and of long units."""
import os
import shutil
import subprocess

import pytest

from oracle import xshare_oracle as O
from paper_2602_07265_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC, INCLUDE = os.path.join(ROOT, "paper_2602_07265_gb300", "csrc"), os.path.join(ROOT, "include")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "pair_rule.cuh"
int main(int argc, char **argv) {
  if (argc == 10) {
    int a[9];
    for (int i = 0; i < 9; ++i) a[i] = std::atoi(argv[1 + i]);
    std::printf("%d\n", xs::selected_at_most(a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8]));
    return 0;
  }
  int v[7];
  for (int i = 0; i < 7; ++i) v[i] = std::atoi(argv[1 + i]);
  std::puts(xs::pair_rule(v[0], v[1], v[2], v[3] != 0, v[4], v[5], v[6]) ? "1" : "0");
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("pair_rule")
    (d / "rule.cpp").write_text(MAIN)
    exe = d / "rule"
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-I" + INCLUDE, str(d / "rule.cpp"), "-o", str(exe)], check=True)
    return exe


@pytest.fixture(scope="module")
def rule(exe):
    def run(T, N, d, F, here=None, sure=True, P=76):
        args = [T * N, N, N if here is None else here, int(sure), P, d, F]
        return subprocess.run([str(exe)] + [str(a) for a in args], capture_output=True, text=True,
                              check=True).stdout.strip() == "1"
    return run


@pytest.mark.parametrize("T,N,d,F,pairs", [
    # Several rounds of units whose last one leaves the pairs idle for long.
    (24, 16, 5120, 2048, False), (32, 16, 5120, 2048, False), (48, 16, 5120, 2048, True),
    (24, 300, 640, 1920, False), (32, 300, 640, 1920, False), (64, 300, 640, 1920, True),
    (24, 16, 6144, 1408, False), (32, 16, 6144, 1408, False), (48, 16, 6144, 1408, True),
    (24, 16, 7168, 2048, False), (64, 16, 7168, 2048, True),
    # As long a wait, but of a wide layer's work.
    (25, 40, 7168, 2048, True), (32, 64, 7168, 2048, True),
    # One round of long units on few SMs: a loss at 24 tokens, a gain at 32.
    (24, 4, 7168, 256, False), (32, 4, 7168, 256, True), (24, 8, 7168, 256, True),
    # Few or narrow experts that gain.
    (24, 8, 2048, 256, True), (24, 4, 2048, 2048, True), (24, 8, 7168, 1024, True), (24, 32, 2048, 256, True),
    (24, 64, 1024, 512, True), (24, 64, 2048, 1024, True), (24, 32, 7168, 2048, True), (24, 5, 1280, 640, True),
    # Below 24 tokens: by the share of idle time.
    (12, 64, 2048, 1024, True), (8, 64, 2048, 1024, False), (16, 128, 2048, 768, False),
    (5, 48, 7168, 2048, False), (6, 120, 7168, 2048, True)])
def test_side_that_measured_faster(rule, T, N, d, F, pairs):
    assert rule(T, N, d, F) == pairs


def test_a_rank_counts_its_own_units(rule):
    # 55 experts of 16 blocks fill whole rounds on one GPU; a rank's seven do not.
    assert rule(8, 55, 7168, 2048) and not rule(8, 55, 7168, 2048, here=7)
    # Plain top-k uses every expert of a rank; of a selection's share the count is a guess.
    assert rule(16, 256, 7168, 2048, here=32) and rule(8, 256, 7168, 2048, here=32)
    assert not rule(8, 256, 7168, 2048, here=32, sure=False)
    assert not rule(64, 8, 2048, 256, P=0)   # the kernels cannot run


@pytest.mark.parametrize("mode,kw,exact", [
    (W.MODE_BATCH, dict(budget=10), True), (W.MODE_BATCH, dict(budget=10, k0=1), False),
    (W.MODE_GROUP, dict(n_groups=8, m_g=3), True), (W.MODE_GROUP, dict(n_groups=4, m_g=20), True),
    (W.MODE_GROUP, dict(n_groups=8, m_g=3, k0=1), False), (W.MODE_HIER, dict(m_r=3, tokens_per_request=4), False),
    (W.MODE_HIER, dict(m_r=2, tokens_per_request=4, k0=1, budget=5), False), (W.MODE_TOPK, {}, True)])
def test_bound_on_the_selected_set(exe, mode, kw, exact):
    """The bound holds on the oracle's selection, and is met where nothing but
    the budget decides."""
    B, N = 12, 64
    full = dict(budget=0, k0=0, m_r=0, tokens_per_request=1, n_groups=1, m_g=0)
    full.update(kw)
    args = [mode, B, N, full["budget"], full["k0"], full["tokens_per_request"], full["m_r"], full["n_groups"],
            full["m_g"]]
    bound = int(subprocess.run([str(exe)] + [str(a) for a in args], capture_output=True, text=True,
                               check=True).stdout)
    sizes = []
    for seed in range(4):
        p = W.random_scores(B, N, seed=seed)
        params = {k: v for k, v in full.items() if k != "budget"}
        sizes.append(O.route(p, 4, full["budget"], mode, **params)["n_selected"])
    assert max(sizes) <= bound
    assert not exact or set(sizes) == {bound}
