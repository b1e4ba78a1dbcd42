"""The walk round the faces of a Voronoi cell (csrc/face_walk.cuh), compiled for
the host: a cube and a cube with cut corners are walked completely; a plane with
two cycles (a pinched face), a stale table entry and a cycle that does not come
back are refused."""
import re
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_0901_4107_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <vector>
#define __host__
#define __device__
#define __forceinline__ inline
%s
using namespace amm::vor;
typedef unsigned T;
static T tri(int a, int b, int c) { return a | b << 8 | c << 16; }
// walks every plane as the kernel does; 1 complete, 0 refused
static int cell(const std::vector<T>& v, unsigned char fill, unsigned long long dead = 0) {
  static unsigned char next[64][64];
  unsigned t[64];
  std::memset(next, fill, sizeof next);
  std::memset(t, 0, sizeof t);
  int start[64], n = 0, walked = 0;
  for (int& s : start) s = 64;
  for (int i = 0; i < (int)v.size(); i++) {
    t[i] = v[i];
    if (dead >> i & 1) continue;
    n++;
    const int p[3] = {(int)(v[i] & 255), (int)(v[i] >> 8 & 255), (int)(v[i] >> 16 & 255)};
    for (int z = 0; z < 3; z++) {
      next[p[z]][p[(z + 1) %% 3]] = (unsigned char)i;
      if (i < start[p[z]]) start[p[z]] = i;
    }
  }
  for (int k = 0; k < 64; k++) {
    if (start[k] == 64) continue;
    int seen = 1;
    const int m = walk_face(k, start[k], t, next, 48, [&](int q) { return q < (int)v.size() && !(dead >> q & 1); },
                            [&](int) { seen++; });
    if (m < 0) return 0;
    if (m != seen) return -1;
    walked += m;
  }
  return walks_complete(walked, n) ? 1 : 0;
}
int main() {
  // a box: planes +x -x +y -y +z -z = 0..5
  std::vector<T> box;
  for (int c = 0; c < 8; c++) {
    const int a = c & 1, b = 2 + (c >> 1 & 1), d = 4 + (c >> 2);
    const bool pos = !((c ^ c >> 1 ^ c >> 2) & 1);
    box.push_back(pos ? tri(a, b, d) : tri(b, a, d));
  }
  int bad = 0;
  for (int fill : {0, 3, 255}) bad += cell(box, (unsigned char)fill) != 1;
  // corner 0 (planes 0, 2, 4) cut by plane 6
  std::vector<T> cut = box;
  cut.push_back(tri(0, 2, 6));
  cut.push_back(tri(2, 4, 6));
  cut.push_back(tri(4, 0, 6));
  for (int fill : {0, 3, 255}) bad += cell(cut, (unsigned char)fill, 1) != 1;
  bad += cell(cut, 0, 2) != 0;                  // an open cell
  // two tetrahedra that share plane 0: it has two cycles
  std::vector<T> two = {tri(0, 1, 2), tri(0, 2, 3), tri(0, 3, 1), tri(1, 3, 2),
                        tri(0, 4, 5), tri(0, 5, 6), tri(0, 6, 4), tri(4, 6, 5)};
  bad += cell(two, 255) != 0;
  bad += cell(std::vector<T>(two.begin(), two.begin() + 4), 255) != 1;
  // plane 0's second vertex leads into a cycle without the first: 0 -> 1 -> 2 -> 1 ...
  bad += cell({tri(0, 1, 2), tri(0, 2, 3), tri(0, 3, 2)}, 255) != 0;
  std::printf("%%d\n", bad);
}
"""


def test_walks(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "walk.cpp"
    src.write_text(MAIN % re.sub(r"(?m)^#pragma.*$", "", (CSRC / "face_walk.cuh").read_text()))
    exe = tmp_path / "walk"
    subprocess.run([gxx, "-O1", "-std=c++17", "-o", str(exe), str(src)], check=True)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) == 0
    assert "walks_complete(" in (CSRC / "voronoi.cu").read_text()
