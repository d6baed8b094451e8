"""Positions in the sliced matrices DF and P_0 (padded rows) at the ends of their 32-bit words.

Matrices of that size take tens of GB on the host, so the rule itself is compiled and run: entries up to
2^31 - 1 and padded entries up to 2^32 - 1 are accepted, one more of either is refused, and a position
comes back from its word as it was."""
import subprocess

CODE = r"""
#include "nls_internal.h"
#include <cstdio>
using namespace nls;
static bool refused(int64_t entries, int64_t padded) {
  try {
    check_sliced(entries, padded, "matrix");
  } catch (const std::runtime_error&) {
    return true;
  }
  return false;
}
int main() {
  const int64_t e = INT32_MAX, p = UINT32_MAX;
  bool ok = !refused(e, p) && !refused(0, 0) && refused(e + 1, e + 1) && refused(1, p + 1);
  for (int64_t at : {int64_t(0), e, e + 1, p}) ok = ok && (int64_t)(uint32_t)position32(at) == at;
  std::puts(ok ? "ok" : "wrong");
}
"""


def test_position_words(tmp_path):
    from paper_2410_24138_gb300 import build
    src = tmp_path / "positions.cpp"
    src.write_text(CODE)
    exe = str(tmp_path / "positions")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True).stdout.strip() == "ok"

