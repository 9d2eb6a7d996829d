"""The choice of a launch's cluster on a GPU (or a partition of one) that has
no room for it: smaller clusters, then none, never an error."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("fit") / "fit")
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_1505_01348_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "cluster_fit_fake.cpp"), "-o", exe], check=True)
    return lambda want, room: int(subprocess.run([exe, str(want), str(room)], check=True, capture_output=True,
                                                 text=True).stdout)


@pytest.mark.parametrize("want,room,got", [(8, 16, 8), (8, 8, 8), (8, 7, 4), (8, 3, 2), (8, 1, 1), (8, 0, 1),
                                           (8, -1, 1), (4, 8, 4), (1, 0, 1), (1, 8, 1)])
def test_cluster_that_fits(choose, want, room, got):
    assert choose(want, room) == got
