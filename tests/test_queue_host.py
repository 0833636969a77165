"""The queue of a batch's registrations (rf_queue.hpp, the code that the kernel
runs), on host threads: whatever the members' delays and however few polls a
member waits, every stream is either registered by all members of exactly one
group, or by none and then reported exactly once; with patient members, all
streams are registered."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_02082_gb300", "csrc")

DRIVER = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>
#include "rf_queue.hpp"
struct Mem {
  std::vector<std::atomic<int>>* abandoned;
  unsigned load(unsigned* p) { return std::atomic_ref<unsigned>(*p).load(std::memory_order_relaxed); }
  unsigned add(unsigned* p, unsigned v) { return std::atomic_ref<unsigned>(*p).fetch_add(v, std::memory_order_relaxed); }
  unsigned cas(unsigned* p, unsigned expected, unsigned v) {
    std::atomic_ref<unsigned>(*p).compare_exchange_strong(expected, v, std::memory_order_relaxed);
    return expected;
  }
  void pause(long long) { std::this_thread::yield(); }
  void abandon(int at) { (*abandoned)[at]++; }
};
int main(int, char** argv) {
  const int n = std::atoi(argv[1]), groups = std::atoi(argv[2]), G = std::atoi(argv[3]);
  const long long limit = std::atoll(argv[4]);
  long whole = 0, reported = 0, wrong = 0;
  for (int trial = 0; trial < 60; ++trial) {
    std::vector<unsigned> links(n, rf::kLinkNone);
    unsigned counter = groups, left = groups;
    std::vector<std::atomic<int>> abandoned(n);
    std::vector<std::vector<std::atomic<int>>> members(n);  // per stream and group
    for (auto& m : members) m = std::vector<std::atomic<int>>(groups);
    std::vector<std::thread> threads;
    for (int g = 0; g < groups; ++g)
      for (int lb = 0; lb < G; ++lb)
        threads.emplace_back([&, g, lb, trial] {
          std::mt19937 rng(trial * 1009 + g * 31 + lb);
          Mem mem{&abandoned};
          for (int at = g; at < n;) {
            members[at][g]++;
            if (rng() % 4 == 0) std::this_thread::sleep_for(std::chrono::microseconds(rng() % 60));
            at = lb == 0 ? rf::queue_lead(mem, links.data(), &counter, &left, at, n)
                         : rf::queue_follow(mem, links.data(), at, n, limit);
          }
        });
    for (auto& t : threads) t.join();
    for (int at = 0; at < n; ++at) {
      int full = 0, none = 0;
      for (int g = 0; g < groups; ++g) {
        full += members[at][g] == G;
        none += members[at][g] == 0;
      }
      const int a = abandoned[at];
      if (full == 1 && none == groups - 1 && a == 0) ++whole;
      else if (none == groups && a == 1) ++reported;
      else ++wrong;
    }
  }
  std::printf("%ld %ld %ld\n", whole, reported, wrong);
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    d = tmp_path_factory.mktemp("queue")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run(["g++", "-O1", "-std=c++20", "-pthread", "-I", CSRC, str(d / "driver.cpp"), "-o", str(exe)],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("n,groups,members", [(1, 1, 3), (7, 2, 3), (12, 3, 2), (5, 5, 2), (9, 1, 1)])
@pytest.mark.parametrize("limit", [0, 1, 8, 10**9])
def test_each_stream_has_one_whole_group_or_is_reported(driver, n, groups, members, limit):
    out = subprocess.run([driver, str(n), str(groups), str(members), str(limit)], capture_output=True, text=True,
                         check=True, timeout=120).stdout
    whole, reported, wrong = map(int, out.split())
    assert wrong == 0
    assert whole >= 60 * groups  # a group always registers its first stream
    assert whole + reported == 60 * n
    if limit == 10**9:
        assert reported == 0
