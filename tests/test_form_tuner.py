"""The choice of a launch form by timing: one disturbed sweep does not decide it, whichever sweep it is, a state that
slows down while it settles does not favour what is tried first, and no more sweeps are taken than programs allow for
(24 for a context's twelve forms, 48 for a batch's eighteen or for eight under the global schedule)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "crmc_tune.h"
// argv: candidates, settling, the best candidate, the disturbed sweep (-1 none), slowing per sweep
int main(int, char **a) {
  const int n = std::atoi(a[1]), best = std::atoi(a[3]), bad = std::atoi(a[4]);
  const float slow = (float)std::atof(a[5]);
  crmc::FormTuner t;
  std::vector<int> c;
  for (int i = 0; i < n; ++i) c.push_back(10 + i);
  t.begin(c, std::atoi(a[2]) != 0);
  int k = 0;
  while (t.on) {
    float ms = t.current() == 10 + best ? 1.0f : 1.1f + 0.01f * (float)(t.current() - 10);
    ms *= 1.0f + slow * (float)(k < 12 ? k : 12);
    if (k == bad) ms *= 20.0f;
    t.record(ms);
    ++k;
  }
  std::printf("%d %d\n", k, t.begun() ? t.current() - 10 : -1);
}
"""


@pytest.fixture(scope="module")
def tuner(tmp_path_factory):
    d = tmp_path_factory.mktemp("tuner")
    (d / "t.cpp").write_text(SOURCE)
    exe = str(d / "t")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2109_07527_gb300", "csrc"),
                           str(d / "t.cpp"), "-o", exe])
    return lambda *a: tuple(int(x) for x in subprocess.check_output([exe] + [str(x) for x in a]).split())


@pytest.mark.parametrize("n,settling,limit", [(12, 0, 24), (18, 0, 48), (10, 0, 25), (5, 0, 25), (8, 1, 48), (4, 1, 24)])
def test_one_disturbed_sweep_does_not_decide(tuner, n, settling, limit):
    for best in (0, n // 2, n - 1):
        sweeps, choice = tuner(n, settling, best, -1, 0.0)
        assert choice == best and sweeps <= limit
        first = n if not settling else 3 * n
        for bad in range(first, sweeps):  # in every counted round
            assert tuner(n, settling, best, bad, 0.0) == (sweeps, best)
        for bad in range(first):  # in the first rounds: the best form or, if it was the one disturbed, one close to it
            assert tuner(n, settling, best, bad, 0.0)[1] in (best, 0, 1)


@pytest.mark.parametrize("n", [4, 8])
def test_a_settling_state_favours_no_form(tuner, n):
    for best in range(n):
        assert tuner(n, 1, best, -1, 0.2)[1] == best


def test_few_candidates(tuner):
    assert tuner(0, 0, 0, -1, 0.0) == (0, -1)
    assert tuner(1, 0, 0, -1, 0.0)[1] == 0
    assert tuner(2, 0, 1, -1, 0.0)[1] == 1
