"""The grid barrier's arrival test (csrc/cr_grid_bar.cuh), compiled with g++: CTAs pass a
barrier when all have arrived and not before, also where the 32-bit counter of
arrivals wraps."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1808_05510_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not found")
    d = tmp_path_factory.mktemp("bar")
    src = d / "bar.cpp"
    src.write_text('#include "cr_grid_bar.cuh"\n'
                   'extern "C" int reached(unsigned v, unsigned t) { return cr::grid_bar_reached(v, t); }\n')
    out = d / "libbar.so"
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", CSRC, "-o", str(out), str(src)], check=True)
    so = C.CDLL(str(out))
    so.reached.argtypes = [C.c_uint, C.c_uint]
    return so


@pytest.mark.parametrize("ctas", [1, 7, 152, 304])
def test_no_barrier_is_passed_early(lib, ctas):
    for k in [1, 2, 2 ** 31 // ctas, 2 ** 32 // ctas, 2 ** 32 // ctas + 1, 2 ** 33 // ctas + 1]:
        for total in (k * ctas, (k + 1) * ctas):  # this barrier and the next
            target = total % 2 ** 32
            for arrived in {0, 1, ctas // 2, ctas - 1}:  # of this barrier's CTAs
                assert bool(lib.reached((total - ctas + arrived) % 2 ** 32, target)) == (arrived == ctas)
            for ahead in {0, 1, ctas - 1}:  # others already at the next barrier
                assert lib.reached((total + ahead) % 2 ** 32, target)
