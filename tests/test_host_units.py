"""Host code of the library compiled on its own: what a device would make awkward to test."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SMEM_PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
#include "kernel_smem.h"
// the two runtime calls, with the limit of one kernel
static std::atomic<int> limit{0}, calls{0};
extern "C" cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
  calls++;
  std::this_thread::sleep_for(std::chrono::microseconds(rand() % 50));
  limit = v;
  return cudaSuccess;
}
int main() {
  static int kernel;
  std::atomic<int> bad{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 8; t++)
    threads.emplace_back([&, t] {
      for (int k = 0; k < 400; k++) {
        const size_t want = 1024 + (size_t)((k * 8 + t) * 7919 % 200000);
        if (amp::allow_dynamic_smem(&kernel, want) != cudaSuccess || limit < (int)want) bad++;      // a launch with `want` bytes would fail
      }
    });
  for (auto& t : threads) t.join();
  printf("%d %d\n", (int)bad, (int)calls);
}
"""


def test_shared_memory_limit_of_a_kernel_is_never_lowered_by_another_thread(tmp_path):
    """Eight threads that launch one kernel with different sizes: at no launch is the kernel's limit below what that launch needs."""
    (tmp_path / "smem.cpp").write_text(SMEM_PROGRAM)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I", os.path.join(cuda, "include"), "-I", os.path.join(ROOT, "paper_1705_09786_b200", "csrc"),
                           str(tmp_path / "smem.cpp"), "-o", str(tmp_path / "smem")])
    bad, calls = (int(v) for v in subprocess.check_output([str(tmp_path / "smem")], text=True, timeout=60).split())
    assert bad == 0 and 1 <= calls < 200


def test_a_newer_file_of_the_sources_or_headers_is_a_reason_to_build(monkeypatch, tmp_path):
    """Every quoted include of the sources is among the files whose time the build looks at."""
    import re

    from paper_1705_09786_b200 import build
    csrc = os.path.dirname(build.SRC)
    deps = {os.path.realpath(d) for d in build.DEPS}
    for f in os.listdir(csrc):
        assert os.path.realpath(os.path.join(csrc, f)) in deps
        for inc in re.findall(r'#include "([^"]+)"', open(os.path.join(csrc, f)).read()):
            assert os.path.realpath(os.path.join(csrc, inc)) in deps, (f, inc)
    lib, dep = tmp_path / "lib.so", tmp_path / "wave_host.cuh"
    lib.write_text("")
    dep.write_text("")
    monkeypatch.setattr(build, "LIB", str(lib))
    monkeypatch.setattr(build, "DEPS", [str(dep)])
    os.utime(lib, (1000, 1000))
    os.utime(dep, (900, 900))
    assert build.up_to_date()
    os.utime(dep, (1100, 1100))
    assert not build.up_to_date()
