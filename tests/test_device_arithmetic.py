"""Index arithmetic of the device code that can be evaluated by the compiler: a translation unit
of static assertions over csrc/agile_dev.cuh (no GPU)."""
import os
import subprocess

from paper_2504_19365_gb300 import build

CHECKS = r"""
#include "agile.h"
#include "agile_dev.cuh"
using agile::requests_a_step;
constexpr bool steps_ok(uint64_t n, uint32_t warps, uint32_t part) {
  const uint32_t t = requests_a_step(n, warps, part);
  // a step moves a warp on, is whole parts, and all warps' steps are enough for n or full
  return t >= part && t <= 32 && t % part == 0 && (t == 32 / part * part || (uint64_t)t * warps >= n);
}
constexpr bool all_ok() {
  const uint64_t ns[] = {1, 2, 3, 31, 32, 33, 2047, 2048, 2049, 65536, 1ull << 31, 0xFFFFF800ull, 0xFFFFF801ull,
                         0xFFFFFFFEull, 0xFFFFFFFFull};
  const uint32_t ws[] = {1, 2, 7, 8, 15, 85, 256, 2047, 2048, 2128, 3072, 65536};
  const uint32_t ps[] = {1, 2, 4, 8, 16, 32};
  for (uint64_t n : ns)
    for (uint32_t w : ws)
      for (uint32_t p : ps)
        if (!steps_ok(n, w, p)) return false;
  return true;
}
static_assert(all_ok(), "requests_a_step");
static_assert(requests_a_step(0xFFFFFFFFull, 2048, 2) == 32, "no wrap at the largest request count");
static_assert(requests_a_step(8192, 2048, 2) == 4, "requests are shared by all warps");
"""


def test_static_assertions(tmp_path):
    src = tmp_path / "checks.cu"
    src.write_text(CHECKS)
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-cubin", "-I", build.INC, "-I", build.CSRC, str(src), "-o",
           os.fspath(tmp_path / "checks.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
