"""The record of dynamic shared memory granted to kernels (csrc/rmt_smem.h), compiled on the host: a grant is a kernel's
on one device, so a second device of a process is granted its own, and it only grows."""
import os
import subprocess

from paper_2104_00095_gb300 import build as B

SRC = r"""
#include "rmt_smem.h"
#include <cstdio>
int main() {
  SmemGrants g;
  int a = 0, b = 0;
  auto ask = [&](int dev, const void* k, size_t bytes, int fail) {
    int calls = 0;
    const int e = g.grant(dev, k, bytes, [&] { calls++; return fail; });
    std::printf("%d%d ", e, calls);
  };
  ask(0, &a, 60000, 0);  // granted
  ask(0, &a, 50000, 0);  // enough already
  ask(1, &a, 60000, 0);  // the other device
  ask(0, &b, 60000, 0);  // the other kernel
  ask(0, &a, 70000, 3);  // refused: not remembered
  ask(0, &a, 70000, 0);
  ask(0, &a, 70000, 0);
  return 0;
}
"""


def test_grants_are_per_device_and_kernel(tmp_path):
    src = tmp_path / "grants.cpp"
    src.write_text(SRC)
    exe = str(tmp_path / "grants")
    subprocess.run(["g++", "-std=c++17", "-I", B.CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["01", "00", "01", "01", "31", "01", "00"]


def test_solvers_opt_in_through_the_record():
    """Every opt-in of the multigrid solvers goes through the record; none is remembered for the process."""
    text = open(os.path.join(B.CSRC, "rmt_mg.cu")).read()
    assert text.count("grants.grant(dev, fn") == 1
    assert text.count("cudaFuncSetAttribute") == 2 and "static size_t" not in text
