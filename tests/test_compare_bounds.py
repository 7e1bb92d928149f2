"""The chunks that the probe's byte comparison reads (loopbounds.h), compiled for the
host with g++: for every alignment of the two keys and every short length, and for
keys up to the longest that count in 32 bits, exactly the R chunks that hold a byte
of the R key are read, each where the S chunk over it needs it, and no count wraps."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HDR = os.path.join(os.path.dirname(HERE), "paper_2411_18183_gb300", "csrc", "loopbounds.h")

PROG = r"""
#include <cstdio>
#include "%s"
using namespace algsig;
typedef unsigned long long u64;
int main() {
  u64 bad = 0, checked = 0;
  auto check = [&](unsigned sa, unsigned d, unsigned len) {
    const u64 end = (u64)sa + len, rlo = sa + d, rend = end + d;     // 64-bit truth; R bytes [rlo, rend)
    const unsigned kend = narrow_end(sa, len), nfull = kend >> 4, rem = kend & 15u;
    if (kend != end || (u64)nfull * 16 + rem != end) bad++;
    auto holds = [&](u64 chunk) { return 16 * chunk < rend && 16 * chunk + 16 > rlo; };
    auto whole = [&](u64 c) {
      if (r_low((unsigned)c, sa, d) != holds(c) || r_high((unsigned)c, nfull, rem, d) != holds(c + 1)) bad++;
    };
    for (u64 c = 0; c < nfull && c < 40; c++) whole(c);
    for (u64 c = nfull > 40 ? nfull - 40 : 0; c < nfull; c++) whole(c);
    if (rem && (r_low_partial(nfull, sa, d) != holds(nfull) || r_high_partial(rem, d) != holds((u64)nfull + 1))) bad++;
    // the first chunk past the last that a trip may count to (two chunks per lane of a warp ahead)
    if ((u64)nfull + 2 * 32 + 256 > 0xFFFFFFFFull || (u64)(unsigned)((nfull << 4) + 16u) != (u64)nfull * 16 + 16) bad++;
    checked++;
  };
  for (unsigned sa = 0; sa < 16; sa++)
    for (unsigned d = 0; d < 16; d++) {
      for (unsigned len = 1; len <= 400; len++) check(sa, d, len);
      for (unsigned k = 1; k <= 300; k++) check(sa, d, kNarrowLen - k);
    }
  printf("%%llu %%llu\n", checked, bad);
  return 0;
}
"""


def test_chunks_read(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = tmp_path / "cb.cpp"
    src.write_text(PROG % HDR)
    exe = tmp_path / "cb"
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-o", str(exe), str(src)])
    checked, bad = map(int, subprocess.check_output([str(exe)]).split())
    assert checked == 256 * 700 and bad == 0
