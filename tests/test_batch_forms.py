"""The kernel form of a batch's launches: the rule by number of (tile, matrix) pairs, and what the autotuner
found where it applies. A form timed at one batch size holds at another one only where the rule gives
the same answer for both: the faster form changes with the number of pairs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "plan.h"
using namespace sym;
static int bad = 0;
static void check(bool ok, const char *what, int kind, int stored, int tuned, int nb) {
  if (!ok) { std::printf("%s kind %d stored %d tuned %d nb %d\n", what, kind, stored, tuned, nb); bad = 1; }
}
int main() {
  const int kinds[4] = {K_UPDATE, K_POTRF, K_TRSM, K_TRTRI};
  const int64_t limit[4] = {BATCH_WARP_UPDATE, BATCH_CTA_POTRF, BATCH_CTA_TRSM, BATCH_CTA_TRTRI};
  for (int i = 0; i < 4; ++i) {
    Launch L = {};
    L.kind = kinds[i];
    L.tb = SMALL_TILE;
    L.count = 17;
    const int few = (int)(limit[i] / L.count), many = few + 1;  // the last batch at the limit, the first beyond
    for (int f64 = 0; f64 < 2; ++f64) {
      const bool flips = f64 || L.kind != K_UPDATE;
      check(batch_default_form(L, 2, false, many, f64) == flips, "rule beyond", L.kind, -1, 0, many);
      check(!batch_default_form(L, 2, false, few, f64), "rule at", L.kind, -1, 0, few);
      for (int nb : {2, few, many, 4 * many})
        for (int tuned : {2, few, many, 4 * many})
          for (int stored = -1; stored < 2; ++stored) {
            const bool rule = batch_default_form(L, 2, false, nb, f64);
            const bool same = rule == batch_default_form(L, 2, false, tuned, f64);
            const bool want = stored < 0 || !same ? rule : stored == 1;
            check(batch_form(L, 2, false, nb, f64, stored, tuned) == want, "form", L.kind, stored, tuned, nb);
          }
    }
    // a warp at 512 matrices, timed there, says nothing about 20
    if (L.kind != K_POTRF) check(!batch_form(L, 2, false, 20, true, 1, 512), "512 to 20", L.kind, 1, 512, 20);
    L.tb = 0;  // full tiles: only updates with small entries have the rule
    check(batch_default_form(L, 0, true, 1000, true) == (L.kind == K_UPDATE), "full tiles", L.kind, -1, 0, 1000);
    check(!batch_default_form(L, 0, false, 1000, true), "large entries", L.kind, -1, 0, 1000);
  }
  PanelForm pf = {PANEL_FUSED, 200, 8, 0};
  for (int nb : {2, 30, 1000})
    for (int tuned : {2, 30, 1000})
      for (int stored = -1; stored < 2; ++stored) {
        const bool rule = batch_level_apart(pf, 5, nb, false);
        const bool want = stored < 0 || batch_level_apart(pf, 5, tuned, false) != rule ? rule : stored == 1;
        check(batch_apart(pf, 5, nb, false, stored, tuned) == want, "apart", 0, stored, tuned, nb);
      }
  return bad;
}
"""


def test_forms_by_batch_size(tmp_path):
    cc = shutil.which("g++")
    if not cc:
        pytest.skip("no C++ compiler")
    src = tmp_path / "forms.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "forms")
    subprocess.run([cc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1705_06575_gb300", "csrc"), str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
