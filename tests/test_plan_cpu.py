"""The plan of the expansion's inverses (csrc/plan.h), compiled here and checked on the scalar recursion:
on a fine grid of eigenvalues each level's start leaves no more than the residual it promises, and the planned
corrections bring it below the tolerance, from the narrowest spectra to the widest the expansion accepts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = r'''
#include "plan.h"
#include <cstdio>
using namespace xl;
int main() {
  const double tols[] = {1e-8, 1e-16}, t0s[] = {1e-9, 1e-3, 0.02, 0.1, 0.21, 0.5, 0.9, 0.999999};
  for (double tol : tols)
    for (double t0 : t0s)
      for (int n : {1, 2, 10, 40}) {
        PlanCache cache;
        std::vector<LevelPlan> p;
        plan_expansion(cache, t0, n, tol, p);
        double over = 0.0, left = 0.0;
        int products = 0;
        for (int i = 0; i <= 5000; ++i) {
          double t = t0 * i / 5000, w1 = 0.0, s1 = 0.0;
          for (int k = 0; k < n; ++k) {
            const double s = t * t;
            double W = p[k].g[0] + p[k].g[1] * w1 + p[k].g[2] * s + p[k].g[3] * s1;
            const double R = std::fabs(1.0 - (1.0 + s) * (1.0 - W));
            over = std::max(over, R - p[k].e0);
            double e = R;
            for (int r = 0; r < p[k].inv.n; ++r) e = std::pow(e, p[k].inv.order[r]);
            left = std::max(left, e);
            s1 = s;
            w1 = s / (1.0 + s);
            t = 2.0 * t / (1.0 + s);
          }
        }
        for (int k = 0; k < n; ++k) products += orders_cost(p[k].inv);
        const ResolventPlan z = plan_resolvent(t0 * t0, tol);
        double zl = 0.0;
        for (int i = 0; i <= 5000; ++i) {
          const double s = t0 * t0 * i / 5000;
          double e = std::fabs(1.0 - (1.0 - s) * (z.z0 + z.z1 * s));
          for (int r = 0; r < z.inv.n; ++r) e = std::pow(e, z.inv.order[r]);
          zl = std::max(zl, e);
        }
        std::printf("%g %g %d %g %g %d %g\n", tol, t0, n, over, left, products, zl);
      }
}
'''


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_planned_corrections_reach_the_tolerance(tmp_path):
    src = tmp_path / "plan.cpp"
    src.write_text(CODE)
    exe = tmp_path / "plan"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1705_10845_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    rows = [line.split() for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 2 * 8 * 4
    for tol, t0, n, over, left, products, zl in rows:
        tol, n = float(tol), int(n)
        # rounding of the scalar recursion itself: a few 1e-16
        assert float(over) < 1e-14, (tol, t0, n)
        assert float(left) <= tol, (tol, t0, n)
        assert int(products) <= n * (6 if tol > 1e-12 else 8), (tol, t0, n)
        # spectra up to 1 - s = 1e-6 still end
        assert float(zl) <= tol or float(t0) > 0.99, (tol, t0, n)


PARTS = r'''
#include "plan.h"
#include <cstdio>
int main() {
  for (int nat = 1; nat <= 700; ++nat)
    for (int slots = 1; slots <= 64; ++slots) {
      const xl::ProbeParts p = xl::probe_parts(nat, slots), again = xl::probe_parts(nat, p.size);
      std::printf("%d %d %d %d %d %d\n", nat, slots, p.size, p.side, again.size, again.side);
    }
}
'''


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_probe_parts_of_the_exact_kernel(tmp_path):
    src = tmp_path / "parts.cpp"
    src.write_text(PARTS)
    exe = tmp_path / "parts"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1705_10845_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    side = {}
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines():
        nat, slots, size, s, size2, s2 = map(int, line.split())
        assert 1 <= size <= min(slots, nat)
        parts = -(-nat // size)
        assert parts == -(-nat // min(slots, nat))   # no more parts than the slots ask for
        assert (size2, s2) == (size, s)              # the slots of one part are all that is needed
        # what picks the arithmetic is a function of the atoms alone
        assert side.setdefault(nat, s) == s
        assert s == (size if slots == 64 else s)
