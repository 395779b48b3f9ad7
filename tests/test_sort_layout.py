"""Sizes of the radix sorts (csrc/sort_layout.h), checked on the CPU by a small C++ program: a
scratch laid out for n items must hold that of every sort of fewer, since one workspace serves all
chunks of a sweep."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_08174_gb300", "csrc")


def run_program(tmp_path, body: str) -> None:
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "check.cpp", tmp_path / "check"
    src.write_text('#include "sort_layout.h"\n#include <cstdio>\nusing namespace ocgs::sort_layout;\n'
                   "int main() {\n" + body + "  return 0;\n}\n")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_scratch_of_n_items_holds_every_smaller_sort(tmp_path):
    """Every n through both tile sizes, then the sizes of records and pairs up to the limit."""
    run_program(tmp_path, """
  const struct { int passes, bits; } plans[] = {{4, 8}, {1, 4}, {2, 7}, {3, 8}};
  for (auto p : plans) {
    size_t most = 0;  // bytes of the largest sort so far
    for (uint64_t n = 0; n < 4000000; ++n) {
      most = std::max(most, bytes_used((uint32_t)n, p.passes, p.bits));
      if (bytes_for((uint32_t)n, p.passes, p.bits) < most) {
        std::printf("n %llu: %zu bytes, a smaller sort uses %zu\\n", (unsigned long long)n,
                    bytes_for((uint32_t)n, p.passes, p.bits), most);
        return 1;
      }
    }
    for (uint64_t n = 4000000; n <= 0xffffffffull; n += 999983) {
      most = std::max(most, bytes_used((uint32_t)n, p.passes, p.bits));
      if (bytes_for((uint32_t)n, p.passes, p.bits) < most) return 1;
    }
  }
""")


@pytest.mark.parametrize("n,views", [(20_000, 20), (20_000, 27), (50_000, 20), (15_000, 31)])
def test_last_chunk_fits_the_workspace_of_the_first(tmp_path, n, views):
    """Depth-sort scratch of a sweep of more than 16 views: chunks of 16, a shorter last one."""
    run_program(tmp_path, f"  return bytes_for({16 * n}u, 4, 8) < bytes_used({(views - 16) * n}u, 4, 8);\n")


def test_digit_plan_covers_every_key_width(tmp_path):
    run_program(tmp_path, """
  for (int n = 1; n <= 32; ++n) {
    const DigitPlan p = digit_plan(n);
    if (p.passes * p.bits < n || p.bits < kMinDigit || p.bits > kMaxDigit || p.passes != (n + 7) / 8) return 1;
  }
""")
