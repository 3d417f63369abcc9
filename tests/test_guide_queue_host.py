"""The tile queue of the guidance distances, on CPU: the functions that the
kernel runs (sfm_guide_queue.h), an atomic operation at a time, under a
scheduler that holds CTAs up between any two of them.  No entry is lost and no
wait is circular, whatever the number of tiles and CTAs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("guide") / "model")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I",
                    os.path.join(ROOT, "paper_1803_04782_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "guide_queue_model.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 6, 9, 40])
@pytest.mark.parametrize("ctas", [1, 2, 5, 12])
def test_no_entry_is_lost_when_ctas_are_held_up(model, tiles, ctas):
    for seed in range(12):
        for hold in (0, 60, 3000):
            r = subprocess.run([model, str(tiles), str(ctas), str(seed), str(hold)], capture_output=True,
                               text=True)
            assert r.returncode == 0, (tiles, ctas, seed, hold, r.stdout)
