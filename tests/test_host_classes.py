"""Class partitions of cells, macro elements and vertex patches
(csrc/host_mesh.cpp) on the CPU, against their definitions.

Two cells share stored matrices when they have the same boundary faces and the
same wavespeed bits; macro elements when their eight children do, place by
place; vertex patches when the eight cells around the vertex do (missing ones
alike).  Members of a patch class have equally many DOFs under both rules.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_01728_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include "host_mesh.h"
using namespace dpgmg;
static void put(const char* name, const std::vector<int32_t>& v) {
  printf("%s", name);
  for (int32_t x : v) printf(" %d", x);
  printf("\n");
}
int main(int argc, char** argv) {
  int n[3] = {atoi(argv[1]), atoi(argv[2]), atoi(argv[3])};
  double a[3] = {0, 0, 0}, b[3] = {1, 1, 1};
  MeshL m;
  m.init(n, 2, a, b);
  std::vector<double> c;
  for (int i = 4; i < argc; ++i) c.push_back(atof(argv[i]));
  const std::vector<int32_t> el = element_classes(m, c);
  put("cells", el);
  put("patches", patch_classes(n, el));
  std::vector<char> sm(m.ndof, 1);
  for (int r2 = 0; r2 < 2; ++r2) {
    std::vector<int32_t> s;
    for (int64_t v : patch_sizes(m, false, 2, n, r2 != 0)) s.push_back((int32_t)v);
    put(r2 ? "sizes2" : "sizes1", s);
  }
  if (n[0] % 2 == 0 && n[1] % 2 == 0 && n[2] % 2 == 0) put("macro", macro_classes(n, el));
  return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("classes")
    (d / "driver.cpp").write_text(DRIVER)
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(d / "driver.cpp"),
                    os.path.join(CSRC, "host_mesh.cpp"), "-o", str(d / "driver")], check=True)
    return str(d / "driver")


def same_partition(ids, keys):
    """ids number the distinct keys in order of first appearance."""
    first = {}
    return all(first.setdefault(k, len(first)) == i for i, k in zip(ids, keys))


@pytest.mark.parametrize("n", [(1, 1, 1), (2, 2, 2), (3, 5, 4), (6, 4, 8), (1, 7, 2)])
@pytest.mark.parametrize("field", ["one", "layers", "random"])
def test_classes_match_their_definitions(driver, n, field):
    nel = n[0] * n[1] * n[2]
    rng = np.random.default_rng(nel)
    c = {"one": np.ones(nel), "layers": np.repeat(rng.choice([0.5, 0.25, 1.0], n[2]), n[0] * n[1]),
         "random": rng.choice([0.5, 1.0], nel)}[field]
    out = subprocess.run([driver, *map(str, n), *("%.17g" % x for x in c)], check=True, capture_output=True, text=True)
    got = {ln.split()[0]: [int(x) for x in ln.split()[1:]] for ln in out.stdout.splitlines()}
    cell = {}
    e = 0
    for k in range(n[2]):
        for j in range(n[1]):
            for i in range(n[0]):
                cell[i, j, k] = (i == 0, i == n[0] - 1, j == 0, j == n[1] - 1, k == 0, k == n[2] - 1, c[e])
                e += 1
    assert same_partition(got["cells"], list(cell.values()))

    def around(i, j, k):
        return tuple(cell.get((i - 1 + (o & 1), j - 1 + (o >> 1 & 1), k - 1 + (o >> 2))) for o in range(8))
    keys = [around(i, j, k) for k in range(n[2] + 1) for j in range(n[1] + 1) for i in range(n[0] + 1)]
    assert same_partition(got["patches"], keys)
    for sizes in (got["sizes1"], got["sizes2"]):
        of = {}
        assert all(of.setdefault(q, s) == s for q, s in zip(got["patches"], sizes))
    if all(x % 2 == 0 for x in n):
        keys = [tuple(cell[2 * i + (o & 1), 2 * j + (o >> 1 & 1), 2 * k + (o >> 2)] for o in range(8))
                for k in range(n[2] // 2) for j in range(n[1] // 2) for i in range(n[0] // 2)]
        assert same_partition(got["macro"], keys)
