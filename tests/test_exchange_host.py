"""The registration's arrival and exit counts (rf_exchange.hpp, the calls that
the kernel makes) in a host model of weakly ordered memory: a relaxed reduction
may take effect at any time up to its thread's next release.  The last CTA to
leave then resets the arrival count, and no arrival may follow the reset.  With
an exit that releases nothing the model shows late arrivals."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_02082_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <utility>
#include <vector>
#include "rf_exchange.hpp"
struct Mem {  // one thread's view: reductions that have not taken effect yet
  bool release;
  std::vector<std::pair<unsigned*, unsigned>> held;
  void flush(size_t keep) {
    for (; held.size() > keep; held.pop_back()) *held.back().first += held.back().second;
  }
  void red_relaxed(unsigned* p, unsigned v) { held.push_back({p, v}); }
  unsigned add_acq_rel(unsigned* p, unsigned v) {
    if (release) flush(0);
    const unsigned old = *p;
    *p += v;
    return old;
  }
};
int main(int, char** argv) {
  const int G = std::atoi(argv[1]), evals = std::atoi(argv[2]);
  const bool release = std::atoi(argv[3]) != 0;
  long late = 0;
  for (int trial = 0; trial < 200; ++trial) {
    std::mt19937 rng(trial);
    unsigned arrivals = 0, left = 0;
    std::vector<Mem> cta(G, Mem{release, {}});
    for (int e = 0; e < evals; ++e)
      for (auto& m : cta) {
        rf::arrive(m, &arrivals);
        if (rng() % 2) m.flush(0);
      }
    for (auto& m : cta)
      if (rf::last_to_leave(m, &left, G)) arrivals = left = 0;
    for (auto& m : cta) m.flush(0);
    late += arrivals != 0 || left != 0;
  }
  std::printf("%ld\n", late);
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("exchange")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(d / "driver.cpp"), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("ctas,evals", [(1, 1), (2, 3), (64, 12), (152, 23)])
def test_no_arrival_follows_the_reset(driver, ctas, evals):
    def late(release):
        return int(subprocess.run([driver, str(ctas), str(evals), str(release)], capture_output=True, text=True,
                                  check=True).stdout)
    assert late(1) == 0
    assert late(0) > 0  # (the model's control)
