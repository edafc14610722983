"""The split of a launch's last tiles into set groups (csrc/tile_split.h) on the CPU: the least cost over
every number of groups, found without trying them all."""
import ctypes
import os
import random
import subprocess
import time

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2406_01821_gb300", "csrc")


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("split") / "libsplit.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC,
                           os.path.join(HERE, "split_cases.cpp"), "-o", so])
    f = ctypes.CDLL(so).split_groups
    f.restype, f.argtypes = ctypes.c_int64, [ctypes.c_int64] * 5
    return f


def every(rest, slots, P, W, base):
    best, groups = None, 1
    for g in range(1, max(1, -(-P // W)) + 1 if rest else 1):
        sets = -(-P // g)
        cost = -(-rest * g // slots) * (base + -(-sets // W) * W)
        if best is None or cost < best:
            best, groups = cost, g
    return groups


@pytest.mark.parametrize("seed", range(4))
def test_equals_the_search_over_all_groups(split, seed):
    rng = random.Random(seed)
    for _ in range(1500):
        slots = rng.choice([1, 2, 152, 304, 456, rng.randint(1, 1000)])
        rest = rng.randint(0, slots - 1)
        W = rng.choice([8, 16, 32])
        P = rng.choice([1, W, W + 1, 64, rng.randint(1, 300), int(2 ** rng.uniform(0, 13))])
        base = 64 + rng.randint(1, 300) // 3
        assert split(rest, slots, P, W, base) == every(rest, slots, P, W, base), (rest, slots, P, W, base)


def test_large_populations_take_no_search(split):
    """A population of 2^31 - 1 sets: trying every number of groups would take minutes."""
    t = time.perf_counter()
    for rest in (1, 151, 152, 303):
        g = split(rest, 304, 2 ** 31 - 1, 16, 74)
        assert 1 <= g and rest * g < 2 ** 31
    assert time.perf_counter() - t < 1.0
