"""Where a key ends in the signature kernel's blocks and steps (loopbounds.h), compiled
for the host with g++: the chunks that are copied around a key's end, its last chunk
and the bytes of it, against 64-bit arithmetic, for short keys at every start and for
keys around 4, 64 and 128 GiB (a key of 64 GiB has 2^32 chunks of 16 bytes)."""
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
  auto check = [&](unsigned a, u64 len) {
    const u64 chunks = (a + len + 15) / 16;
    const KeyEnd e = key_end(a, len);
    if (e.blocks != (chunks + 1) / 2 || e.rest != (a + len) %% 16) bad++;
    if (8ull * last_step(e.blocks) + last_place(e.blocks, e.full) != chunks - 1) bad++;
    for (u64 c = chunks > 40 ? chunks - 40 : 0; c < chunks + 40; c++)
      if (has_chunk((unsigned)(c / 8), c %% 8, c %% 2 ? e.full : e.blocks) != (c < chunks)) bad++;
    if (!has_chunk(0, 0, e.blocks)) bad++;
    checked++;
  };
  for (unsigned a = 0; a < 32; a++)
    for (u64 len = 1; len <= 600; len++) check(a, len);
  const u64 tops[] = {1ull << 32, 1ull << 36, (1ull << 37) - 2000};
  for (u64 top : tops)
    for (unsigned a = 0; a < 32; a++)
      for (u64 len = top - 300; len <= top + 300; len++) check(a, len);
  for (unsigned q = 0; q < 8; q++)
    if (has_chunk(0, q, 0)) bad++;                     // an empty key has none
  printf("%%llu %%llu\n", checked, bad);
  return 0;
}
"""


def test_key_end(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src = tmp_path / "ke.cpp"
    src.write_text(PROG % HDR)
    exe = tmp_path / "ke"
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-o", str(exe), str(src)])
    checked, bad = map(int, subprocess.check_output([str(exe)]).split())
    assert checked > 70_000 and bad == 0
