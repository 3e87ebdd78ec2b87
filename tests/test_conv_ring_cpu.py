"""The tensor-core router's two converter groups on its ring of stages, on the CPU.

conv_ring.cuh is compiled for the host and run against a model of the kernel's
barriers (parity waits, as the hardware answers them), its TMA loads (which may
land in any order) and its MMAs.  Every schedule must convert the bytes of the
step it is meant to, and the MMAs must find the planes of their step.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_07265_gb300", "csrc")

MODEL = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "conv_ring.cuh"

constexpr int kGroups = 2;

struct Bar {  // one arrival per phase; a wait on parity p passes if the last completed phase has it
  int done = 0;
  bool passes(uint32_t parity) const { return ((done & 1) ^ 1) == static_cast<int>(parity); }
};

// Runs `steps` steps over `stages` stages.  late >= 0: the load of that step
// lands only when nothing else can move; else the order is drawn from `seed`.
// Returns the first fault: a step number, -1 for none, -2 for a standstill.
int run(int stages, int steps, int late, unsigned seed, bool full_only) {
  std::vector<Bar> full(stages), conv(stages), empty(stages);
  std::vector<int> loaded(stages, -1), planes(stages, -1);
  std::vector<int> flight;                                  // loads on their way
  std::vector<xs::ConvRing<kGroups>> ring;
  std::vector<int> at;                                      // next step of each group
  for (int g = 0; g < kGroups; ++g) ring.emplace_back(g, stages), at.push_back(g);
  int issued = 0, multiplied = 0, released = 0;
  std::mt19937 rng(seed);
  while (released < steps) {
    std::vector<int> can;                                   // enabled moves
    if (issued < steps && empty[issued % stages].passes(((issued / stages) & 1) ^ 1)) can.push_back(0);
    for (size_t i = 0; i < flight.size(); ++i)
      if (flight[i] != late) can.push_back(100 + static_cast<int>(i));
    for (int g = 0; g < kGroups; ++g)
      if (at[g] < steps &&
          ring[g].wait([&](int s, uint32_t p) { return full_only || empty[s].passes(p); },
                       [&](int s, uint32_t p) { return full[s].passes(p); }))
        can.push_back(10 + g);
    if (multiplied < steps && conv[multiplied % stages].passes((multiplied / stages) & 1)) can.push_back(1);
    if (released < multiplied) can.push_back(2);
    if (can.empty()) {
      if (flight.empty()) return -2;
      can.push_back(100);                                   // the late load is the only one left
      for (size_t i = 0; i < flight.size(); ++i)
        if (flight[i] == late) can[0] = 100 + static_cast<int>(i);
    }
    const int m = can[rng() % can.size()];
    if (m == 0) {
      flight.push_back(issued++);
    } else if (m == 1) {
      if (planes[multiplied % stages] != multiplied) return multiplied;
      ++multiplied;
    } else if (m == 2) {
      ++empty[released % stages].done;
      ++released;
    } else if (m >= 100) {
      const int k = flight[m - 100];
      flight.erase(flight.begin() + (m - 100));
      loaded[k % stages] = k;
      ++full[k % stages].done;
    } else {
      const int g = m - 10, k = at[g], s = ring[g].stage;
      if (s != k % stages || loaded[s] != k) return k;
      planes[s] = k;
      ++conv[s].done;
      ring[g].next();
      at[g] += kGroups;
    }
  }
  return -1;
}

int main(int argc, char **argv) {
  const int stages = std::atoi(argv[1]);
  const bool full_only = std::atoi(argv[2]) != 0;
  for (int steps : {1, 2, stages, 2 * stages + 1, 29})
    for (unsigned seed = 0; seed < 60; ++seed)
      for (int late = -1; late < steps; ++late) {
        const int bad = run(stages, steps, late, seed, full_only);
        if (bad != -1) {
          std::printf("stages %d steps %d late %d seed %u: fault at step %d\n", stages, steps, late, seed, bad);
          return 1;
        }
      }
  return 0;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("conv_ring")
    (d / "model.cpp").write_text(MODEL)
    exe = d / "model"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + CSRC, str(d / "model.cpp"), "-o", str(exe)], check=True)
    return exe


# 3, 5 and 6 stages are what 64, 32 and 16 experts per tile get.
@pytest.mark.parametrize("stages", [2, 3, 4, 5, 6])
def test_every_step_is_converted_from_its_own_load(model, stages):
    r = subprocess.run([str(model), str(stages), "0"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("stages", [3, 5])
def test_the_model_finds_a_group_that_waits_for_the_load_alone(model, stages):
    r = subprocess.run([str(model), str(stages), "1"], capture_output=True, text=True, timeout=120)
    assert r.returncode == 1 and "fault" in r.stdout
