"""The adaptive rule's rate test: lambda is lowered when Delta d^T Delta d
changes by less than `ratio` per sweep, for every ratio > 0 -- down to one that
only a residual that no longer changes at all passes."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rate_rule_against_its_definition(tmp_path):
    # csrc/wf_rate.h against |1 - q^(1/R)| < ratio in extended precision, for q
    # around both bounds, at 1 and at the ends of the range.  Left out: q whose
    # rate is within 1e-9 of ratio or, in q, within two units of the last place
    # (2^-52 / R in the rate) -- there rounding decides.
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "rate.cpp"
    src.write_text(r'''
#include <cmath>
#include <initializer_list>
#include <cstdio>
#include "wf_rate.h"
int main() {
  int bad = 0, n = 0;
  const int Rs[] = {1, 2, 10, 50, 1000};
  for (int R : Rs)
    for (double e = -20; e <= 2.01; e += 0.125) {
      const double ratio = std::pow(10.0, e);
      const wf::RateBounds b = wf::rate_bounds(ratio, R);
      double qs[64];
      int nq = 0;
      for (double f : {0.0, 0.3, 0.9, 0.999, 1.001, 1.1, 3.0, 100.0})
        for (double s : {-1.0, 1.0})
          if (s * f * ratio > -1.0) qs[nq++] = (double)expl(R * log1pl((long double)(s * f * ratio)));
      for (double q : {1.0, std::nextafter(1.0, 0.0), std::nextafter(1.0, 2.0), 0.5, std::nextafter(0.5, 0.0), 2.0,
                       1e-30, 1e-300, 1e30, 1e300}) qs[nq++] = q;
      for (int i = 0; i < nq; ++i) {
        const double q = qs[i];
        if (!(q > 0.0) || std::isinf(q)) continue;
        const long double rate = fabsl(expm1l(logl((long double)q) / R));
        if (q != 1.0 && fabsl(rate - ratio) < 1e-9L * ratio + 4.5e-16L / R * fmaxl(1.0L, rate)) continue;
        ++n;
        if (wf::rate_below(b, q) != (rate < ratio)) {
          std::printf("R %d ratio %.17g q %.17g rate %.17Lg\n", R, ratio, q, rate);
          ++bad;
        }
      }
      if (wf::rate_below(b, HUGE_VAL) || wf::rate_below(b, NAN)) ++bad;
    }
  return bad || n < 5000;
}
''')
    exe = tmp_path / "rate"
    inc = os.path.join(ROOT, "paper_1704_00865_gb300", "csrc")
    r = subprocess.run([cxx, "-std=c++17", "-I", inc, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]


@pytest.mark.gpu
@pytest.mark.parametrize("ratio", [1e-17, 1e-16, 1e-12])
def test_lambda_falls_once_the_residual_stands_still(ratio):
    # at lambda = 5e5 the white-noise iteration is at its FP32 fixed point after
    # a few sweeps: two checkpoints of a level with the same residual, bit for
    # bit, pass any ratio, so the next one runs at lambda^0.7
    from gpu_util import make_plan
    from paper_1704_00865_gb300 import build, synth, wf
    build.build()
    wf.load()
    prob = synth.make_problem(64, 64, 3, one_over_f=False, stripes=False, mask_frac=0.0)
    plan = make_plan(prob, residual_every=10, max_iters=200, trace=1)
    plan.run(wf.make_schedule("adaptive", lam0=5e5, ratio=ratio, expo=0.7), 0.0)
    t = plan.trace()
    plan.close()
    still = [i for i in range(1, len(t) - 1)
             if t[i]["lam"] == t[i - 1]["lam"] > 1.0 and t[i]["rel_rho_u"] == t[i - 1]["rel_rho_u"]]
    assert len(t) == 20 and still
    for i in still:
        assert t[i + 1]["lam"] == pytest.approx(t[i]["lam"] ** 0.7, rel=1e-12), i
