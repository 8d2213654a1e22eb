"""The rules of fe_rules.cuh, compiled for the host, against times measured on a GB300 (152 SMs):
at each measured size the kernel that a rule chooses is at most 3 % (and 0.2 us) slower than
the fastest one measured there.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

from _util import ROOT

SMS = 152

HARNESS = r"""
#include "fe_rules.cuh"
extern "C" int four_case_passes(long n, int R, int sms) { return fe::four_case_passes(n, R, sms); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("rules")
    (d / "r.cpp").write_text(HARNESS)
    so = str(d / "r.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fPIC", "-shared", str(d / "r.cpp"), "-o", so,
                    "-I", os.path.join(ROOT, "paper_1710_08679_gb300", "csrc")], check=True)
    return ctypes.CDLL(so)


def near_best(chosen, times):
    return times[chosen] <= 1.03 * min(times.values()) + 0.2


# us per inner step at level 0: one case per thread, four cases per thread
@pytest.mark.parametrize("n,R,one,four", [
    (1331, 4, 24.0, 26.1), (1331, 32, 26.3, 27.2), (1331, 64, 29.7, 29.0), (4913, 8, 25.7, 26.1),
    (4913, 16, 28.6, 29.1), (4913, 20, 33.9, 31.5), (4913, 64, 67.4, 50.8), (9261, 4, 25.5, 27.1),
    (9261, 8, 28.6, 29.1), (9261, 12, 32.5, 31.9), (15625, 4, 28.0, 29.1), (15625, 8, 35.9, 34.4),
    (24389, 4, 31.1, 31.0), (205757, 16, 263.4, 252.8)])
def test_passes_of_four_cases(rules, n, R, one, four):
    assert near_best(rules.four_case_passes(ctypes.c_long(n), R, SMS), {0: one, 1: four})


@pytest.mark.parametrize("R", [1, 2, 6, 13])
def test_passes_of_four_cases_need_a_multiple_of_four(rules, R):
    assert not rules.four_case_passes(ctypes.c_long(10**7), R, SMS)
