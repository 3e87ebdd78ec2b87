"""The rule between the two routers (router_rule.cuh), on the CPU: the side
that measured faster on GB300, over widths, batches and expert counts."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_07265_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "router_rule.cuh"
int main(int, char **argv) {
  std::puts(xs::router_on_tensor_cores(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[3])) ? "1" : "0");
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("router_rule")
    (d / "rule.cpp").write_text(MAIN)
    exe = d / "rule"
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(d / "rule.cpp"), "-o", str(exe)], check=True)
    return lambda B, N, d: subprocess.run([str(exe), str(B), str(N), str(d)], capture_output=True, text=True,
                                          check=True).stdout.strip() == "1"


@pytest.mark.parametrize("B,N,d,tensor", [
    (63, 1024, 8192, False), (64, 8, 4096, True), (150, 64, 2048, False), (250, 64, 2048, False),
    (350, 64, 2048, True), (992, 32, 1024, True), (512, 32, 1024, False),
    # Narrow layers with many logits: small d, but the CUDA cores lose up to 70 %.
    (1984, 128, 128, True), (512, 128, 128, True), (248, 1024, 128, True), (4096, 32, 128, True),
    (992, 128, 256, True), (3072, 32, 256, True), (496, 128, 512, True), (7936, 8, 512, True),
    (128, 128, 256, False), (512, 32, 256, False), (128, 128, 512, False), (2048, 8, 512, False)])
def test_side_that_measured_faster(rule, B, N, d, tensor):
    assert rule(B, N, d) == tensor
