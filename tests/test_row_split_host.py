"""The row kernel's hand-out of strips, played through on the host (no GPU): `row_split_model.cpp` with the kernel's own arithmetic."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("split") / "model")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2505_18573_b200", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "row_split_model.cpp")], check=True)
    return exe


def _play(model, *args):
    r = subprocess.run([model, *map(str, args)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.parametrize("slow", [4, 14, 400])
@pytest.mark.parametrize("rows, tiles, sampler, cta", [
    (4608, 75, -1, 2), (4096, 75, 1, 15), (1200, 75, 1, -1), (4096, 250, 0, 2)])  # a short segment one ring before a longer one
def test_state_of_a_segment_is_not_shared(model, rows, tiles, sampler, cta, slow):
    _play(model, rows, tiles, sampler, 148, slow, cta, 1)


@pytest.mark.parametrize("slow", [4, 400])
@pytest.mark.parametrize("rows, tiles, sampler, cta", [
    (300, 977, 1, 0), (1000, 600, 1, 0), (1000, 600, 1, 6),   # pieces of two to four half rings, one behind the other
    (900, 1040, -1, 5), (700, 2100, -1, 3), (400, 6500, 0, 2)])
def test_state_of_a_long_piece_is_not_shared(model, rows, tiles, sampler, cta, slow):
    _play(model, rows, tiles, sampler, 148, slow, cta, 3)


@pytest.mark.parametrize("rows, tiles, sampler", [(4096, 75, -1), (6144, 75, 0), (512, 75, 1), (2000, 125, 1), (900, 333, -1)])
def test_every_block_finishes(model, rows, tiles, sampler):
    _play(model, rows, tiles, sampler, 148, 60, -1, 41)
