"""Opting in to more than 48 KB of dynamic shared memory (csrc/dwf_optin.h) without a GPU: per
device, the largest size so far, again after a failure; compiled with g++."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_0423_gb300", "csrc")

PROG = r'''
#include <cstdio>
#include <thread>
#include <vector>
#include "dwf_optin.h"
using namespace dwf;
int main() {
  SmemOptIn k;
  int calls = 0;
  auto at = [&](int dev, size_t kb, int rc) {
    const int before = calls, e = k.ensure(dev, kb * 1024, [&] { ++calls; return rc; });
    printf("%d:%zu %d %d\n", dev, kb, calls - before, e);
  };
  at(0, 48, 0);   // needs none
  at(0, 60, 0);   // the first
  at(0, 60, 0);   // known
  at(0, 52, 0);   // less
  at(1, 60, 0);   // another device
  at(0, 90, 1);   // larger, refused
  at(0, 90, 0);   // so asked again
  at(1, 90, 0);
  at(0, 90, 0);
  SmemOptIn t;
  int n = 0;
  std::vector<std::thread> th;
  for (int i = 0; i < 8; ++i) th.emplace_back([&, i] { for (int r = 0; r < 100; ++r) t.ensure(i & 3, 65536, [&] { ++n; return 0; }); });
  for (auto &x : th) x.join();
  printf("threads %d\n", n);
}
'''


def test_each_device_is_opted_in_once_per_size(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)])
    out = subprocess.check_output([str(exe)], text=True).splitlines()
    assert out == ["0:48 0 0", "0:60 1 0", "0:60 0 0", "0:52 0 0", "1:60 1 0", "0:90 1 1", "0:90 1 0", "1:90 1 0",
                   "0:90 0 0", "threads 4"]


def test_launchers_take_the_helper():
    """No launcher keeps a size of its own that forgets the device."""
    src = open(os.path.join(CSRC, "dwf_launch.cuh")).read()
    assert src.count("cudaFuncSetAttribute") == 1 and "static size_t" not in src
