"""The autotuner's candidates are distinct launches (CPU; the rules alone, compiled with nvcc).

Width settings (cells per block) are rounded to what a kernel lays out: curved
passes to 512 threads, axis-aligned ones to bricks of cells.  Every candidate has
to be another launch than the others, named by the cells that its blocks take,
and that number as a setting has to give the launch again.
"""
import itertools
import json
import subprocess

import pytest

from paper_1910_01900_gb300 import build
from paper_1910_01900_gb300.csrc_info import max_cells_per_block

MESHES = [(4, 4, 4), (64, 64, 1), (16, 16, 16), (1, 7, 33), (5, 4, 6), (32, 31, 30)]
KEEP = 4
MAIN = r"""
#include <cstdio>
#include "dg_launch.cuh"
#include "fe_box.cuh"
using namespace sipg;
template <typename T>
void run(int n, bool curved, const int (&m)[3]) {
  const int64_t cells = (int64_t)m[0] * m[1] * m[2];
  const int most = max_cb(n, sizeof(T));
  auto launch = [&](int cb) { return dg_tile_launch<T>(n, curved, m, cells, cb); };
  printf("{\"key\": [%d, %d, %d, %d, %d, %d], \"widths\": [", (int)sizeof(T), n, (int)curved, m[0], m[1], m[2]);
  const char *c = "";
  for (int w : pick_widths(0, most, cells, 152, KEEP, launch, [&](const TileLaunch &t) { return 2048 / t.threads; }))
    printf("%s%d", c, w), c = ", ";
  printf("], \"launch\": [");
  c = "";
  for (int cb = 0; cb <= most; ++cb) {
    const TileLaunch t = launch(cb);
    printf("%s[%d, %d, %lld]", c, t.cells, t.threads, (long long)t.blocks), c = ", ";
  }
  printf("]}\n");
}
// FE levels of axis-aligned cells: the default brick, and the one of a width
template <typename T>
void bricks(int n, const int (&m)[3]) {
  printf("{\"key\": [%d, %d, \"fe\", %d, %d, %d], \"bricks\": [", (int)sizeof(T), n, m[0], m[1], m[2]);
  for (int cb = 0; cb <= 512; ++cb) {
    int b[3];
    fe_box_brick<T>(n, m, cb, b);
    const TileLaunch t = fe_box_launch<T>(n, m, b);
    printf("%s[%d, %d, %d, %d]", cb ? ", " : "", b[0], b[1], b[2], t.cells);
  }
  auto launch = [&](int cb) {
    int b[3];
    fe_box_brick<T>(n, m, cb, b);
    return fe_box_launch<T>(n, m, b);
  };
  printf("], \"widths\": [");
  const char *c = "";
  for (int w : pick_widths(launch(0).cells, max_cb(n, sizeof(T)), (int64_t)m[0] * m[1] * m[2], 152, KEEP, launch,
                           [&](const TileLaunch &t) { return 2048 / t.threads; }))
    printf("%s%d", c, w), c = ", ";
  printf("]}\n");
}
int main() {
  const int meshes[][3] = MESHES;
  for (int n = 2; n <= 9; ++n)
    for (auto &m : meshes) bricks<float>(n, m), bricks<double>(n, m);
  for (int n = 2; n <= 9; ++n)
    for (int curved = 0; curved < 2; ++curved)
      for (auto &m : meshes) run<float>(n, curved, m), run<double>(n, curved, m);
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rules")
    src = MAIN.replace("MESHES", "{%s}" % ", ".join("{%d, %d, %d}" % m for m in MESHES)).replace("KEEP", str(KEEP))
    (d / "main.cu").write_text(src)
    subprocess.run([nvcc] + build.ARCH + ["-std=c++17", "-I", build.CSRC, str(d / "main.cu"), "-o", str(d / "main")],
                   check=True, capture_output=True)
    out = subprocess.run([str(d / "main")], check=True, capture_output=True, text=True).stdout
    return {tuple(r["key"]): r for r in map(json.loads, out.splitlines())}


@pytest.mark.parametrize("n,elem,curved", list(itertools.product(range(2, 10), (4, 8), (0, 1))))
def test_candidates_are_distinct_launches(rules, n, elem, curved):
    for m in MESHES:
        r = rules[(elem, n, curved) + m]
        launches = [tuple(t) for t in r["launch"]]   # of the settings 0 (default), 1, 2, ...
        assert len(launches) == max_cells_per_block(n, elem) + 1
        for setting, (cells, threads, blocks) in enumerate(launches):
            assert cells <= max(setting or cells, 2 if elem == 4 and not curved else 1)
            assert threads == cells * n * n // (1 if curved or elem == 8 else 2)
            assert blocks * cells >= m[0] * m[1] * m[2]
            assert launches[cells] == (cells, threads, blocks)
        widths = r["widths"]
        assert widths[0] == launches[0][0]
        assert len(set(launches[w] for w in widths)) == len(widths) == min(KEEP + 1, len(set(launches)))


@pytest.mark.parametrize("n,elem", list(itertools.product(range(2, 10), (4, 8))))
def test_fe_brick_of_a_width(rules, n, elem):
    """A width is the most cells of a brick, and the cells of a brick as a width give the brick again."""
    for m in MESHES:
        bricks = rules[(elem, n, "fe") + m]["bricks"]
        for cb, (b0, b1, b2, cells) in enumerate(bricks):
            assert cells == b0 * b1 * b2 and (cells <= cb or cb == 0)
            assert bricks[cells] == bricks[cb]
        widths = rules[(elem, n, "fe") + m]["widths"]
        settings = [0] + list(range(1, max_cells_per_block(n, elem) + 1))
        assert widths[0] == bricks[0][3]
        assert len(widths) == len(set(widths)) == min(KEEP + 1, len(set(bricks[c][3] for c in settings)))


def test_tuned_widths_of_one_mesh_are_not_another_meshes(tmp_path):
    """Axis-aligned blocks depend on the mesh's sides, curved ones on the number of cells alone."""
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    (tmp_path / "key.cpp").write_text("""
#include "tile_rules.h"
int main() {
  const int a[3] = {64, 64, 1}, b[3] = {16, 16, 16}, c[3] = {1, 64, 64};
  auto key = [](bool curved, const int *m) { return sipg::tune_key(4, curved, 1, 1, 4096, m); };
  const bool ok = key(false, a) != key(false, b) && key(false, a) != key(false, c) && key(false, b) == key(false, b) &&
                  key(true, a) == key(true, b) && key(true, b) != key(false, b);
  return ok ? 0 : 1;
}
""")
    subprocess.run([nvcc, "-std=c++17", "-I", build.CSRC, str(tmp_path / "key.cpp"), "-o", str(tmp_path / "key")],
                   check=True, capture_output=True)
    assert subprocess.run([str(tmp_path / "key")]).returncode == 0
