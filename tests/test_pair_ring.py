"""The barriers of the CTA-pair kernel, in a model that runs its warps in many orders (tests/ring_model.cpp) with the kernel's own turns of
the converters (csrc/turns.h): no wait by parity ends before the phase it means, and none never ends, whichever warp stays behind."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("ring") / "ring_model")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", os.path.join(HERE, "ring_model.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n128,narrow,adapter_stages,tiles,runs,length", [
    (5, 0, 0, 3, 0, 0),               # half a packed tile at the end: one turn of four missing from tile to tile
    (8, 0, 0, 3, 0, 0),               # turns that come out even
    (9, 0, 3, 4, 0, 0), (6, 0, 2, 4, 0, 0), (8, 0, 7, 3, 0, 0),          # adapter stages in between, 1 to 3 turns off
    (4, 0, 1, 5, 2, 3), (32, 0, 7, 3, 1, 6),                             # T' first
    (1, 0, 1, 9, 0, 0), (2, 0, 6, 6, 1, 1),                              # tiles of fewer stages than groups
    (12, 1, 0, 3, 0, 0), (12, 1, 3, 3, 0, 0), (9, 1, 2, 4, 1, 7), (3, 1, 6, 5, 2, 2), (2, 1, 1, 9, 0, 0),      # stages of a whole packed tile
    (0, 0, 5, 3, 1, 4),               # adapters alone
])
def test_every_wait_ends_and_none_too_early(model, n128, narrow, adapter_stages, tiles, runs, length):
    out = subprocess.run([model, *map(str, (n128, narrow, adapter_stages, tiles, runs, length, 400))], capture_output=True, text=True, timeout=120)
    assert out.stdout == "ok\n", out.stdout
