"""The code that a one-launch stage solve leaves in its record, for every way in which its CTAs can end: the
largest of what they report (an expired barrier wait above a non-finite value above the cap)."""
import ctypes
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1512_00616_gb300", "csrc")


@pytest.fixture(scope="module")
def solve_code(tmp_path_factory):
    d = tmp_path_factory.mktemp("record")
    src = d / "record.cpp"
    src.write_text('#include "solve_record.h"\nextern "C" int code(int alive, int flag, int need, int first) '
                   "{ return pp::solve_code(alive != 0, flag, need != 0, first != 0); }\n")
    so = d / "record.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so)).code


@pytest.mark.parametrize("flag", range(5))
@pytest.mark.parametrize("need", [0, 1])
def test_record_of_all_endings(solve_code, flag, need):
    for alive in itertools.product([0, 1], repeat=4):
        rec = max(solve_code(a, flag, need, cta == 0) for cta, a in enumerate(alive))
        if not all(alive):
            assert rec == 8      # whichever CTA expired
        elif flag == 4:
            assert rec == 4
        else:
            assert rec == (1 if need and flag in (0, 3) else 0)
