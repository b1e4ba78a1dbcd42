"""The places of runs in the tessellation's half-face list (csrc/half_list.cuh),
compiled for the host: runs taken one behind the other up to counts past 2^31
and 2^32 (275 M generators of 15.6 half-faces each) lie inside the list and
apart from one another or are refused, and a count past the capacity asks for
a list that holds it."""
import re
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_0901_4107_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include <initializer_list>
#define __host__
#define __device__
%s
using namespace amm::vor;
int main() {
  const int64_t caps[] = {1024, 18ll * 262144 + 1024, 0x7fffffff - 64, 0x80000000ll, 0x180000000ll};
  const int runs[] = {64, 16, 15, 4};
  int bad = 0;
  for (int64_t cap : caps)
    for (int m : runs)
      for (unsigned long long base : {0ull, (unsigned long long)cap - 70, 0x7fffffc0ull, 0xffffffc0ull, 0x1ffffffc0ull}) {
        if (base > (1ull << 40)) continue;
        unsigned long long at = base;
        for (int q = 0; q < 40; q++, at += m) {
          const int64_t p = half_place(at, m, cap);
          bad += p >= 0 ? !(p == (int64_t)at && p + m <= cap) : !(at + m > (unsigned long long)cap);
        }
        const int64_t more = half_more(at, cap);
        bad += at <= (unsigned long long)cap ? more != 0 : more < (int64_t)at;
      }
  std::printf("%%d\n", bad);
}
"""


def test_places_past_32_bits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "half.cpp"
    src.write_text(MAIN % re.sub(r"(?m)^#pragma.*$", "", (CSRC / "half_list.cuh").read_text()))
    exe = tmp_path / "half"
    subprocess.run([gxx, "-O1", "-std=c++17", "-o", str(exe), str(src)], check=True)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) == 0


def test_the_device_counts_in_64_bits():
    text = (CSRC / "voronoi.cu").read_text()
    body = text[text.index("half_room(const HalfList"):]
    body = body[:body.index("\n}\n")]
    assert "atomicAdd(H.used, (unsigned long long)" in body and "half_place(" in body
    assert re.search(r"unsigned long long\* used;\s*int64_t cap;", text)
