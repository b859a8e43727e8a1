"""The choice between forms of a product from timings (csrc/tune.h) on the CPU:
launches disturbed by other work must not decide it, and a choice made beside
other work is not kept before it has been timed again."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_01728_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "tune.h"
using namespace dpgmg;
int main() {
  int forms, reps, alone;
  TuneRecord r;
  while (scanf("%d %d %d", &forms, &reps, &alone) == 3) {
    std::vector<std::vector<float>> t(forms, std::vector<float>(reps));
    for (auto& v : t)
      for (float& x : v)
        if (scanf("%f", &x) != 1) return 1;
    r.add(t, alone != 0);
    printf("%d %d\n", (int)r.best(), (int)r.settled);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("tune")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "driver.cpp"), "-o", str(d / "driver")], check=True)

    def run(*timings):
        text = ""
        for alone, t in timings:
            text += "%d %d %d\n" % (len(t), len(t[0]), alone) + "\n".join(" ".join(map(str, v)) for v in t) + "\n"
        out = subprocess.run([str(d / "driver")], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, ln.split())) for ln in out.splitlines()]
    return run


FAST, SLOW = [24.0] * 5, [78.0] * 5


def test_disturbed_launches_do_not_decide(choose):
    hit = [24.0, 900.0, 24.0, 24.0, 400.0]          # two launches waited for other work
    assert choose((1, [hit, SLOW])) == [(0, 1)]
    assert choose((1, [SLOW, hit])) == [(1, 1)]
    assert choose((1, [[24, 300, 500, 700, 25], SLOW, FAST])) == [(0, 1)]


def test_the_first_form_is_kept_within_five_per_cent(choose):
    assert choose((1, [[100.0] * 5, [96.0] * 5]))[0][0] == 0
    assert choose((1, [[100.0] * 5, [94.0] * 5]))[0][0] == 1
    assert choose((1, [[100.0] * 5, [94.0] * 5, [93.9] * 5]))[0][0] == 2


def test_a_choice_made_beside_other_work_is_timed_again(choose):
    crowded = [[90.0] * 5, [80.0] * 5]              # every launch of the fast form was disturbed
    assert choose((0, crowded), (0, [FAST, SLOW])) == [(1, 0), (0, 0)]
    assert choose((0, crowded), (1, [FAST, SLOW])) == [(1, 0), (0, 1)]
    assert [s for _, s in choose(*[(0, crowded)] * 3)] == [0, 0, 1]
