"""The serving kernel's agreement to leave (csrc/serve_close.h) on the CPU: a CTA that enters and one
that closes the kernel, each run between any two steps of the other."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2406_01821_gb300", "csrc")


@pytest.fixture(scope="module")
def case(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("close") / "libclose.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC,
                           os.path.join(HERE, "close_cases.cpp"), "-o", so])
    return ctypes.CDLL(so).close_case


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("held", [0, 1, 3])
@pytest.mark.parametrize("at", [0, 1, 2, 3, 99])
def test_either_the_kernel_closes_or_a_cta_enters(case, first, held, at):
    r = case(first, held, at)
    closed, entered, marked, count = r & 1, r >> 1 & 1, r >> 2 & 1, r >> 3
    assert closed == marked
    assert closed + entered == 1, "a CTA entered a closed kernel, or neither got through"
    assert entered or held == 0                    # held units keep the kernel open
    assert count == held + entered
