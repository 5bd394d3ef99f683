"""The host model that picks the greedy's cluster size (csrc/gram_schedule.h), compiled with
the host compiler: the same choice as scheduling every request, at a bounded cost."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_27952_gb300", "csrc")

DRIVER = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <queue>
#include <random>
#include "gram_schedule.h"
using namespace last;
// every request, one after another
static double all_of_them(const std::vector<SchedRequest> &r, int c, int active, int warps) {
  std::priority_queue<double, std::vector<double>, std::greater<double>> free;
  for (int i = 0; i < active; ++i) free.push(0.0);
  double end = 0.0;
  for (const SchedRequest &q : r) {
    const int slots = (q.blocks + c * warps - 1) / (c * warps);
    const double t = free.top() + q.rounds * (27.0 + 4.6 * slots + 0.4 * c);
    free.pop();
    free.push(t);
    end = std::max(end, t);
  }
  return end;
}
int main(int argc, char **argv) {
  const int n = atoi(argv[1]), most = atoi(argv[2]), warps = 15;
  for (int seed = 0; seed < 20; ++seed) {
    std::mt19937 g(seed);
    std::vector<SchedRequest> r(n);
    for (auto &q : r) {
      q.blocks = 1 + (int)(g() % most);
      q.rounds = q.blocks * (1 + g() % 8) / 4.0 + 2.0;
    }
    std::sort(r.begin(), r.end(), [](const SchedRequest &a, const SchedRequest &b) { return a.rounds > b.rounds; });
    Schedule s;
    long long asked = 0;
    schedule_begin(&s, n, [&](int i) { ++asked; return r.at(i); });
    int got = 0, want = 0;
    double best = 0.0, true_best = 0.0;
    for (int c = 1; c <= 16; ++c) {
      const int active = std::max(1, 152 / c - c / 4);
      const double end = schedule_end(&s, c, active, warps, got == 0 ? INFINITY : best);
      if (got == 0 || end < best) { got = c; best = end; }
      const double t = all_of_them(r, c, active, warps);
      if (want == 0 || t < true_best) { want = c; true_best = t; }
    }
    const double cost = all_of_them(r, got, std::max(1, 152 / got - got / 4), warps) / true_best;
    printf("%d %d %.4f %lld\n", got, want, cost, asked);
  }
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("schedule")
    (d / "main.cpp").write_text(DRIVER)
    exe = str(d / "main")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,most_blocks", [(1, 512), (7, 60), (64, 18), (128, 128), (300, 500), (1024, 40),
                                           (1025, 40), (5000, 100), (60000, 3), (60000, 500)])
def test_choice(driver, n, most_blocks):
    out = subprocess.run([driver, str(n), str(most_blocks)], check=True, capture_output=True, text=True).stdout
    for line in out.split("\n")[:-1]:
        got, want, cost, asked = line.split()
        assert int(asked) <= 1024                       # whatever the batch
        if n <= 1024:
            assert got == want
        assert float(cost) <= 1.02, line
