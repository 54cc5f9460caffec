"""Blocks that a sweep unit stages, checked on the CPU from the header that the host and the kernel share: every
row copied by a bulk asynchronous copy starts on 16 bytes, is a whole number of 16 bytes long and not empty,
stays inside its row, and covers the entries the unit reads; a front without boundary rows (a root) stages no
off-diagonal block at all."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "sweep.h"
using namespace fdfd;
int bad = 0;
void check(bool ok, const char* what, int es, int sweep, bool rect, int k, int m, int r0, int cnt, int a, int b) {
  if (!ok && bad++ < 10)
    printf("%s: es %d sweep %d rect %d k %d m %d lines %d + %d part %d..%d\n", what, es, sweep, rect, k, m, r0, cnt, a, b);
}
void one(int es, int sweep, bool rect, int k, int m, int r0, int cnt, int a, int b) {
  const int n = k + m, ld = (n + 3) / 4 * 4, ldk = (k + 3) / 4 * 4;
  const StageGeom g = stage_geom(es, sweep, rect, k, ld, ldk, r0, cnt, a, b, 256);
  auto ck = [&](bool ok, const char* what) { check(ok, what, es, sweep, rect, k, m, r0, cnt, a, b); };
  if (cnt <= 0 || b <= a) {
    ck(g.rows == 0 && stage_bytes(g, es) == 0, "nothing to stage");
    return;
  }
  // the entries the products read, in the front or in the inverse block
  const bool by_row = sweep < 2;
  const int i0 = (rect && (sweep == 0 || sweep == 3) ? k : 0) + (by_row ? r0 : a), in = by_row ? cnt : b - a;
  const int j0 = (rect && (sweep == 1 || sweep == 2) ? k : 0) + (by_row ? a : r0), jn = by_row ? b - a : cnt;
  ck(g.row0 == i0 && g.rows == in, "rows");
  ck(g.col0 + g.shift == j0 && g.shift >= 0 && g.col0 + g.cols >= j0 + jn, "columns");
  ck(g.col0 >= 0 && g.col0 + g.cols <= (rect ? ld : ldk) && g.row0 + g.rows <= (rect ? n : k), "inside");
  ck(g.cols > 0 && g.cols * es % 16 == 0 && g.col0 * es % 16 == 0, "16 bytes");
  ck(g.stride >= g.cols && g.stride * es % 16 == 0, "stride");
}
int main() {
  for (int es = 8; es <= 16; es += 8)
    for (int sweep = 0; sweep < 4; ++sweep) {
      const bool up = sweep == 0 || sweep == 2;
      for (int k = 1; k <= 70; ++k)
        for (int m : {0, 1, 2, 3, 5, 8, 31, 64, 97}) {
          one(es, sweep, true, k, m, 0, up ? m : k, 0, up ? k : m);      // a front swept whole
          for (int rect = 0; rect < 2; ++rect) {
            if (rect && m == 0) continue;
            const int len = rect && up ? m : k;
            for (int c : {8, 16, 64})
              for (int s0 = 0; s0 < len; s0 += c) {
                const int cnt = c < len - s0 ? c : len - s0;
                const UnitRange ur = unit_range(sweep, rect, k, m, s0, cnt);
                for (int part : {8, 24, 128})
                  for (int lo = ur.lo; lo < ur.hi; lo += part)
                    one(es, sweep, rect, k, m, s0, cnt, lo, lo + part < ur.hi ? lo + part : ur.hi);
              }
          }
        }
    }
  printf("%d bad\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_staged_blocks(tmp_path):
    src = tmp_path / "geom.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "geom"
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", cuda, "-I",
                        os.path.join(ROOT, "paper_2307_05388_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
