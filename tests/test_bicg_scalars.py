"""The decisions of the resident FP64 BiCGSTAB solve (csrc/bicg_scalars.cuh) on
the host: random solves whose residuals fall, blow up, break down and become
non-finite in either phase, with the iterates as numbers.  The copy of the best
iterate is the one whose residual the blow-up test compares with, and a restart
from the best iterate starts from it.  A solve that met its tolerance, was found
far from it by its true residual and went on ends as met, with an iterate no
worse than the one it was checked at."""
import os
import subprocess

import pytest

from paper_2106_07616_gb300 import _build

MAIN = r"""
#include "bicg_scalars.cuh"
#include <map>
#include <string>
using namespace rbffd;

static unsigned long long seed = 1;
static double u01() {
  seed = seed * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(seed >> 11) / 9007199254740992.0;
}

int main() {
  std::map<std::string, int> n;
  const double inf = 1e308 * 10, tol = 1e-4;
  for (int solve = 0; solve < 20000; ++solve) {
    BicgScalars c;
    bicg_start(c);
    const bool is_long = solve % 2;  // long enough for the true-residual check
    const int maxit = 20 + (int)(180 * u01()) + (is_long ? BICG_CHECK_ITS : 0);
    const double p_s = 0.05 * u01(), p_r = 0.05 * u01(), p_blow = 0.1 * u01(), p_zero = 0.02 * u01();
    std::map<int, double> res;  // squared residual of every iterate
    int x = 0, xb = -1, made = 0;
    double checked = -1.0;  // largest true residual that a check found and went on from
    res[0] = 1.0;
    for (;;) {
      if (c.state == KRY_RUNNING && c.need_init) {
        const bool best = c.restore;
        if (bicg_from_copy(c)) x = xb;
        if (best) {
          n["restores"]++;
          if (res[x] != c.best2) n["not_from_best"]++;
        }
        if (c.met) {
          n["checks"]++;
          if (u01() < 0.7) {
            res[x] *= 1e6;
            if (res[x] > BICG_CHECK2 * c.tol2) checked = fmax(checked, res[x]);
          }
        }
        bicg_restarted(c, 1.0, res[x], tol);
        if (is_long && c.it == 0) c.it = BICG_CHECK_ITS;
      }
      if (c.state != KRY_RUNNING) break;
      const bool first = c.first;
      if (c.save) xb = x;
      if (!first) x = ++made;
      // the iterate just formed: falling, blown up, or no number
      double rr = res[first ? x : x - 1 < 0 ? 0 : x - 1];
      if (!first) {
        rr *= u01() < 0.6 ? (is_long ? 0.2 : 0.5) : 1.6;
        if (u01() < p_blow) rr *= 1e21;
        if (u01() < p_r) rr = inf;
        res[x] = rr;
      }
      bicg_after_v(c, 1.0, rr, 1.0, maxit);
      if (!c.save && c.best2 < 1e308 && (xb < 0 || res[xb] != c.best2)) n["copy_not_best"]++;
      if (c.save && res[x] != c.best2) n["saves_not_best"]++;
      c.run = c.run && c.state == KRY_RUNNING;
      if (!c.run) continue;
      const double ss = u01() < p_s ? inf : rr;
      if (ss == inf) n["non_finite_s"]++;
      bicg_after_t(c, ss, 1.0, 0.5, u01() < p_zero, 0.5, 2.0, 1.0, maxit);
      if (c.half == 1) res[x = ++made] = ss;
    }
    if (c.state == KRY_RUNNING) n["unfinished"]++;
    const int before = c.state;
    if (bicg_end(c)) x = xb;
    if (checked > 0.0) {
      n["went_on"]++;
      if (before != KRY_OK) n["kept"]++;
      if (c.state != KRY_OK || c.rr > c.tol2) n["failed_after_met"]++;
      if (!(res[x] <= checked)) n["worse_than_checked"]++;
    } else if (c.state != before) {
      n["changed_end"]++;
    }
    n["solves"]++;
  }
  for (const char *k : {"solves", "restores", "non_finite_s", "unfinished", "not_from_best",
                        "copy_not_best", "saves_not_best", "checks", "went_on", "kept",
                        "failed_after_met", "worse_than_checked", "changed_end"})
    printf("%s %d\n", k, n[k]);
}
"""


@pytest.fixture(scope="module")
def counts(tmp_path_factory):
    d = tmp_path_factory.mktemp("scalars")
    (d / "walk.cu").write_text(MAIN)
    exe = str(d / "walk")
    subprocess.run(["nvcc", *_build.ARCH, "-std=c++17", "-I", os.path.join(_build.HERE, "csrc"),
                    "-I", _build.INCLUDE, "-o", exe, str(d / "walk.cu")], check=True,
                   capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    return {k: int(v) for k, v in (line.split() for line in out.split("\n") if line)}


def test_a_restart_starts_from_the_best_iterate(counts):
    assert counts["solves"] == 20000 and counts["unfinished"] == 0
    assert counts["restores"] > 1000 and counts["non_finite_s"] > 1000
    assert counts["not_from_best"] == 0
    assert counts["copy_not_best"] == counts["saves_not_best"] == 0


def test_a_solve_that_met_its_tolerance_does_not_fail_after_it(counts):
    assert counts["checks"] > 1000 and counts["went_on"] > 500 and counts["kept"] > 100
    assert counts["failed_after_met"] == counts["worse_than_checked"] == 0
    assert counts["changed_end"] == 0
