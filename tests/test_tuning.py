"""The autotuner's conclusions (csrc/tuning.h), compiled by themselves."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "tuning.h"
#include <cstdio>
#include <cstdlib>
#include <cstring>
using namespace dd4dv;
int main(int argc, char** argv) {
  if (!std::strcmp(argv[1], "ckpt")) {
    for (int k : checkpoint_candidates(std::atoi(argv[2]), std::atoi(argv[3]))) std::printf("%d ", k);
    return 0;
  }
  if (!std::strcmp(argv[1], "box")) {
    std::printf("%d", level_box_fits(std::atoll(argv[2]), std::atoll(argv[3]), std::atoll(argv[4]), std::atoll(argv[5])));
    return 0;
  }
  SweepTimes t[2];
  double* f[8] = {&t[0].cluster_f, &t[0].cluster_a, &t[0].level_f, &t[0].level_a,
                  &t[1].cluster_f, &t[1].cluster_a, &t[1].level_f, &t[1].level_a};
  for (int k = 0; k < 8; ++k)
    if (std::strcmp(argv[4 + k], "-")) *f[k] = std::atof(argv[4 + k]);
  const SweepChoice c = choose_sweeps(t, std::atoi(argv[2]), std::atoi(argv[3]));
  std::printf("%d %d %d %.6g", c.stored, c.level_f, c.level_a, c.ms);
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("tuning")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2205_06649_gb300", "csrc"), str(d / "t.cpp"),
                    "-o", str(d / "t")], check=True)
    return lambda *a: subprocess.run([str(d / "t"), *map(str, a)], check=True, capture_output=True, text=True).stdout


# stages recomputed: cluster forward, adjoint, level forward, adjoint; then stored
@pytest.mark.parametrize("stored,ckpt,ms,want", [
    # 16-step checkpoints (differentiation workload): the level adjoint alone cannot run
    (0, 1, "1.68 4.91 1.72 3.18 - - - -", "0 1 1 4.9"),
    (0, 1, "1.0 4.0 3.5 3.0 - - - -", "0 0 0 5"),       # level forward too dear: clusters for both
    (0, 1, "1.0 2.0 0.8 3.0 - - - -", "0 1 0 2.8"),     # a cluster adjoint may follow a level forward
    (0, 0, "1.68 4.91 1.72 3.18 - - - -", "0 0 1 4.86"),  # every level stored: any pair
    (1, 0, "2 5 2.5 4 2.1 3 2.6 3.5", "1 0 0 5.1"),
    (1, 0, "2 5 2.5 4 2.1 3 2.6 2.5", "1 0 1 4.6"),
    (0, 0, "2 5 - - 1 1 1 1", "0 0 0 7"),               # no stage buffer: its times do not count
    (1, 0, "- - 2 3 - - 1.5 2", "1 1 1 3.5"),           # no cluster shape timed
])
def test_choose_sweeps(run, stored, ckpt, ms, want):
    assert run("sweeps", stored, ckpt, *ms.split()) == want


def test_no_checkpoint_interval_is_timed_where_none_has_an_effect(run):
    assert run("ckpt", 1, 1) == ""
    for f, a in ((0, 0), (1, 0), (0, 1)):
        assert run("ckpt", f, a).split() == ["8", "16", "32"]


def magic_quotient(a, d):
    """mdiv(a, magic_of(d)) of csrc/point.cuh."""
    m = 0 if d <= 1 else (0xFFFFFFFF // d + 1) & 0xFFFFFFFF
    return (a * m) >> 32 if m else a


@pytest.mark.parametrize("nx,ny,v,fits", [
    (179, 85, 4, True), (2048, 1024, 1, False), (1024, 512, 1, True), (1025, 1365, 1, False), (1024, 1365, 1, True),
    (5, 37837, 4, True), (5, 37838, 4, False), (4097, 86, 4, False), (4096, 85, 4, True),
])
def test_level_boxes_whose_quotients_are_exact(run, nx, ny, v, fits):
    nq, nxp = (nx + v - 1) // v, (nx + 3) // 4 * 4
    assert run("box", nx, ny, nxp, nq) == ("1" if fits else "0")
    if fits:
        for n, d in ((nq * ny, nq), (3 * ny * nx, nx), (3 * ny, ny)):
            step = max(1, n // 4001)
            for a in [*range(0, n, step), *range(max(0, n - 3 * d), n, max(1, d // 7)), n - 1, n - d - 1]:
                assert magic_quotient(a, d) == a // d, (a, d)
