"""The streamed forward hands its stage buffers back by barrier parity.  A
model of the protocol with commits arriving in any order: no warp writes into
a buffer whose MMAs may still read it and none waits forever.  One barrier per
buffer, which needs commits in order, fails the same model."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1505_01348_gb300", "csrc")
SIM = os.path.join(ROOT, "tests", "fwd_ring_sim.cpp")
TASKS = [4, 6, 7, 8, 10, 12]        # per stage: 2 x (2 .. 6 chunks), and an odd number


@pytest.fixture(scope="module")
def sim(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    exe = str(tmp_path_factory.mktemp("ring") / "sim")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, SIM, "-o", exe], check=True)
    return lambda *a: subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout.strip()


@pytest.mark.parametrize("ntask", TASKS)
def test_no_buffer_is_written_early(sim, ntask):
    for seed in range(60):
        for stages in (1, 2, 3, 40):
            assert sim(0, stages, ntask, seed) == "ok"


def test_one_barrier_per_buffer_needs_commits_in_order(sim):
    seen = {sim(2, 40, n, seed) for n in TASKS for seed in range(60)}
    assert seen & {"early", "stuck"}
