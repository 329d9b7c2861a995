"""The ring that passes the beam's children between candidate groups, run on the
CPU in many interleavings of its atomic steps (the code the kernels compile):
groups and pushers that stand still between any two steps, groups that leave after
the idle limit, the smallest rings.  No mark is ever taken for an item, no item is
drawn twice, and every shot ends."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2512_07057_gb300", "csrc")


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ring") / "ring_host.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-o", out,
                    os.path.join(HERE, "ring_host.cpp")], check=True)
    lib = C.CDLL(out)
    lib.ring_host.argtypes = [C.c_uint64] + [C.c_int] * 8 + [C.c_long, C.POINTER(C.c_long)]
    return lib.ring_host


@pytest.mark.parametrize("groups,entries,width", [(4, 1, 1), (4, 2, 1), (4, 2, 2), (8, 4, 1), (16, 3, 2), (5, 8, 2)])
@pytest.mark.parametrize("jumps", [0, 6])
@pytest.mark.parametrize("stalls,sleep", [(40, 60), (60, 600)])
def test_every_item_is_drawn_once_and_every_shot_ends(ring, groups, entries, width, jumps, stalls, sleep):
    marks = 0
    for seed in range(1, 13):
        n = C.c_long(0)
        rc = ring(seed, groups, entries, width, 12 * entries, 5, stalls, sleep, jumps, 4_000_000, C.byref(n))
        assert rc == 0, (seed, rc)
        marks += n.value
    assert jumps == 0 or groups < 2 * entries or marks > 0   # groups have left (more of them than the shots keep busy)
