"""The planner keeps a batch in one pass at lx_eri_workspace_size, whatever the forms of its quartets
and the pairs they share, and accepts it one quartet at a time at lx_eri_workspace_min.

Checked on the host: the probe compiles the planner's translation unit and plans without a device."""
import glob
import os
import subprocess

import pytest

from paper_2307_03452_gb300 import build, lx

HERE = os.path.dirname(os.path.abspath(__file__))
SOLID, SPLIT = lx.LX_SOLID, lx.LX_PATH_SPLIT
# l, K, bra pairs, ket pairs, flags, J/K: lists whose pairs many quartets share, in the axial form
# (contracted ones need more for their tables than the shared pairs leave), in the matrix form
# ((pp|pp), and K = 16 on every (dd|dd) shell), on the split path, and of shells of all l or degrees,
# where both forms hold the same pairs
LISTS = [(2, 3, 64, 64, SOLID, 0), (2, 5, 32, 64, SOLID, 0), (2, 5, 32, 32, 0, 0), (2, 5, 32, 32, SOLID, 1),
         (3, 5, 32, 32, SOLID, 0), (4, 5, 32, 32, 0, 1), (4, 2, 16, 48, SOLID, 0), (6, 1, 64, 64, SOLID, 0),
         (7, 3, 8, 8, 0, 0), (1, 5, 40, 40, SOLID, 0), (2, 16, 4, 4, SOLID, 0), (6, 1, 32, 32, SOLID | SPLIT, 0),
         (2, 3, 1, 1, SOLID, 0), (6, 4, 1, 2, SOLID, 1), (-1, -16, 12, 12, SOLID, 0), (2, -16, 12, 12, 0, 1),
         (-1, -5, 24, 24, 0, 0)]


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("planner") / "probe")
    build.build()
    objs = [o for o in glob.glob(os.path.join(build.BUILD, "*.o")) if os.path.basename(o) != "lx_api.cu.o"]
    cmd = [build.nvcc(), *build.ARCH, "-O1", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
           os.path.join(HERE, "planner_probe.cu"), *objs, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    text = "\n".join(" ".join(map(str, x)) for x in LISTS)
    r = subprocess.run([exe], input=text, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rows = [tuple(map(int, line.split())) for line in r.stdout.split("\n") if line]
    assert len(rows) == len(LISTS)
    return dict(zip(LISTS, rows))


@pytest.mark.parametrize("case", LISTS)
def test_one_pass_at_the_workspace_size(case, plans):
    assert plans[case][0] == 1


@pytest.mark.parametrize("case", LISTS)
def test_smaller_workspaces(case, plans):
    _, half, least, below, fits = plans[case]
    nquartet = case[2] * case[3]
    assert fits == 1
    assert 1 <= half <= least <= nquartet  # never an error: one quartet always fits
    assert below == -6                     # LX_ERR_WORKSPACE
