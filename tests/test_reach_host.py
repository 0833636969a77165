"""Which buffers rf_process_frame's staging kernels may use directly (rf_reach.hpp),
with faked pointer attributes: memory of the volume's own device, managed and
wholly page-locked host memory; another device's memory, pageable and partly
registered memory and unknown pointers go to the copy engine."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1905_02082_gb300", "csrc")

DRIVER = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include "rf_reach.hpp"
int main() {
  // page-locked: [4096, 8192), mapped elsewhere: [16384, 20480)
  auto attributes = [](cudaPointerAttributes* at, const void* p) {
    std::memset(at, 0, sizeof(*at));
    const uintptr_t a = (uintptr_t)p;
    at->devicePointer = (void*)p;
    if (a == 1) return cudaErrorInvalidValue;
    if (a >= 4096 && a < 8192) at->type = cudaMemoryTypeHost;
    else if (a >= 16384 && a < 20480) at->type = cudaMemoryTypeHost, at->devicePointer = (void*)(a + (1 << 20));
    else if (a >= (1 << 24) && a < (2 << 24)) at->type = cudaMemoryTypeDevice, at->device = 0;
    else if (a >= (2 << 24) && a < (3 << 24)) at->type = cudaMemoryTypeDevice, at->device = 1;
    else if (a >= (3 << 24)) at->type = cudaMemoryTypeManaged, at->device = 1;
    else at->type = cudaMemoryTypeUnregistered, at->devicePointer = nullptr;
    return cudaSuccess;
  };
  unsigned long long p, bytes;
  int device;
  while (std::scanf("%llu %llu %d", &p, &bytes, &device) == 3)
    std::printf("%d\n", (int)rf::reachable((const void*)(uintptr_t)p, (size_t)bytes, device, attributes));
  return 0;
}
"""

OWN, OTHER, MANAGED = 1 << 24, 2 << 24, 3 << 24
CASES = [((OWN, 1000, 0), 1), ((OTHER, 1000, 0), 0), ((OWN, 1000, 1), 0), ((OTHER, 1000, 1), 1), ((MANAGED, 10, 0), 1),
         ((4096, 4096, 0), 1), ((4097, 1, 1), 1), ((4096, 4097, 0), 0), ((8191, 2, 0), 0), ((8191, 0, 0), 1),
         ((16384, 16, 0), 0), ((30000, 16, 0), 0), ((1, 16, 0), 0)]


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    from paper_1905_02082_gb300.build import nvcc
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    d = tmp_path_factory.mktemp("reach")
    (d / "driver.cpp").write_text(DRIVER)
    exe = d / "driver"
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", include, str(d / "driver.cpp"), "-o", str(exe)],
                   check=True)
    return str(exe)


def test_buffers_that_kernels_may_use(driver):
    text = "".join("%d %d %d\n" % c for c, _ in CASES)
    out = subprocess.run([driver], input=text, capture_output=True, text=True, check=True).stdout
    assert [int(x) for x in out.split()] == [want for _, want in CASES]


ALIGNED = r"""
#include <cstdio>
#include "rf_reach.hpp"
int main() {
  auto attributes = [](cudaPointerAttributes* at, const void* p) {
    *at = cudaPointerAttributes{};
    at->type = cudaMemoryTypeDevice;
    return cudaSuccess;
  };
  for (unsigned long long p = 1 << 20; p < (1 << 20) + 32; ++p) {
    const void* q = (const void*)(uintptr_t)p;
    std::printf("%d %d\n", (int)rf::staged_by_kernel(q, 64, rf::kImageAlign, 0, attributes),
                (int)rf::staged_by_kernel(q, 64, rf::kWordAlign, 0, attributes));
  }
  return 0;
}
"""


def test_unaligned_buffers_go_to_the_copy_engine(tmp_path):
    """The kernels copy images in 16-byte accesses, poses and infos in 8-byte ones."""
    from paper_1905_02082_gb300.build import nvcc
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    (tmp_path / "aligned.cpp").write_text(ALIGNED)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", include, str(tmp_path / "aligned.cpp"), "-o",
                    str(tmp_path / "aligned")], check=True)
    out = subprocess.run([str(tmp_path / "aligned")], capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in out] == [v for p in range(32) for v in (int(p % 16 == 0), int(p % 8 == 0))]
