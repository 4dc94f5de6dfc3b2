"""The volume solver's tile queue (csrc/mf_tile_queue.cuh, the code the kernel runs) on the CPU, under a model of the
GPU's memory order with a seeded scheduler (tile_queue_model.cpp): every queued tile is visited, by one warp at a time,
after what was written before. The model finds each of three mistakes when it is made in its memory operations."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1507_01926_gb300", "csrc")


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("queue") / "model")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "tile_queue_model.cpp"), "-o", exe])

    def run(tiles, warps, visits, seed, mode=0, hold=20000):
        return subprocess.run([exe, *map(str, (tiles, warps, visits, seed, mode, hold))], check=True, capture_output=True,
                              text=True, timeout=120).stdout.strip()

    return run


@pytest.mark.parametrize("tiles,warps", [(1, 8), (2, 8), (3, 5), (7, 8), (40, 16)])
def test_every_tile_is_visited_once_at_a_time_and_in_order(model, tiles, warps):
    for seed in range(8):
        assert model(tiles, warps, 2000, seed) == "ok", seed


@pytest.mark.parametrize("mode,finds", [(1, {"race"}), (2, {"lost", "twice"}), (3, {"twice", "race", "lost"})])
def test_the_model_finds_mistakes(model, mode, finds):
    got = {model(tiles, 8, 2000, seed, mode) for tiles in (2, 7) for seed in range(8)} - {"ok"}
    assert got and got <= finds, got
