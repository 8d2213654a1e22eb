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
extern "C" int direct_two_cases(long n, int R) { return fe::direct_two_cases(n, R); }
extern "C" int level1_two_blocks(long n, int R, int sms) { return fe::level1_two_blocks(n, R, sms); }
extern "C" int f64_direct_split(long n, int R, int sms) { return fe::f64_direct_split(n, R, sms); }
extern "C" int f64_adjoint_split(long n, int R, int sms) { return fe::f64_adjoint_split(n, R, sms); }
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


# us per FP32 direct product with one case and with two cases per thread (to 4 %: between the
# smallest and largest meshes the two are as near to each other as that)
@pytest.mark.parametrize("n_elem,R,one,two", [
    (750, 16, 6.5, 6.4), (3072, 4, 6.7, 6.7), (3072, 24, 10.2, 11.2), (3072, 48, 14.7, 16.0), (7986, 6, 9.6, 9.1),
    (7986, 16, 13.5, 15.5), (7986, 64, 38.6, 40.3), (16464, 2, 10.3, 9.3), (16464, 8, 14.3, 15.4),
    (16464, 18, 28.2, 27.7), (16464, 32, 39.3, 40.3), (31104, 6, 22.4, 20.9), (31104, 16, 38.7, 39.9),
    (31104, 28, 67.5, 64.5), (73728, 2, 22.8, 20.3), (73728, 32, 166.4, 158.4), (146124, 32, 336.1, 315.3)])
def test_cases_per_thread_of_the_fp32_product(rules, n_elem, R, one, two):
    times = {0: one, 1: two}
    assert times[rules.direct_two_cases(ctypes.c_long(n_elem), R)] <= 1.04 * min(one, two)


@pytest.mark.parametrize("R", [1, 3, 7, 31])
def test_two_cases_need_an_even_number(rules, R):
    assert not rules.direct_two_cases(ctypes.c_long(10**6), R)


# us per level-1 product with one and with two blocks of a row in flight
@pytest.mark.parametrize("n,R,one,two", [
    (6825, 64, 8.4, 8.3), (10875, 64, 10.8, 12.6), (14025, 48, 11.2, 12.8), (14025, 56, 13.7, 14.8),
    (14025, 64, 15.0, 14.4), (21793, 64, 19.1, 20.1), (27132, 28, 12.8, 14.8), (27132, 56, 21.8, 23.3),
    (42189, 16, 11.5, 13.3), (42189, 20, 16.4, 16.2), (59625, 32, 30.1, 27.3), (83997, 8, 12.6, 14.1),
    (83997, 20, 32.5, 29.8), (181476, 4, 25.0, 28.6), (181476, 8, 34.9, 35.9), (181476, 12, 46.6, 45.3),
    (181476, 16, 56.1, 52.8), (181476, 64, 176.2, 167.7)])
def test_blocks_in_flight_of_the_level1_product(rules, n, R, one, two):
    assert near_best(rules.level1_two_blocks(ctypes.c_long(n), R, SMS), {0: one, 1: two})


# us per FP64 direct product by lanes per element (0: a lane per corner), the fastest few
@pytest.mark.parametrize("n_elem,R,times", [
    (750, 1, {0: 11.1, 1: 22.9}),
    (750, 48, {48: 41.0, 24: 42.4, 0: 53.3, 16: 56.1, 12: 73.1, 10: 91.8, 8: 107.1}),
    (3072, 1, {0: 11.5, 1: 23.1}),
    (3072, 8, {8: 32.7, 4: 40.2, 0: 40.9, 3: 57.9, 2: 75.1, 1: 140.0}),
    (3072, 12, {12: 41.8, 6: 43.1, 0: 53.4, 4: 56.9, 3: 75.2, 2: 110.3, 1: 207.3}),
    (3072, 24, {12: 73.4, 24: 79.1, 6: 79.9, 8: 84.7, 5: 97.8, 0: 101.7, 4: 107.7}),
    (7986, 9, {9: 79.8, 3: 83.6, 0: 96.0, 2: 99.3, 5: 104.1, 1: 164.7}),
    (7986, 18, {9: 143.8, 18: 151.6, 4: 154.1, 6: 159.3, 3: 160.3, 2: 171.8, 0: 186.5}),
    (16464, 1, {1: 25.8, 0: 27.0}),
    (16464, 9, {9: 152.3, 2: 155.1, 3: 159.9, 1: 172.2, 5: 178.3, 0: 192.5}),
    (31104, 9, {3: 264.6, 1: 277.6, 9: 279.5, 5: 283.9, 2: 338.2, 0: 356.0}),
    (50544, 5, {5: 245.3, 1: 265.7, 3: 282.9, 2: 309.7, 0: 320.1}),
    (73728, 16, {2: 1060.7, 8: 1068.0, 1: 1070.6, 4: 1070.7, 16: 1115.2, 6: 1169.3, 3: 1192.4}),
    (146124, 5, {1: 676.6, 5: 698.1, 2: 795.5, 3: 795.5}),
    (146124, 30, {5: 3751.6, 3: 3761.9, 6: 3767.5, 10: 3805.3, 2: 3826.1, 15: 3877.0, 1: 3928.4})])
def test_lanes_of_the_fp64_product(rules, n_elem, R, times):
    assert near_best(rules.f64_direct_split(ctypes.c_long(n_elem), R, SMS), times)


# us per sensitivity pass by lanes per element
@pytest.mark.parametrize("n_elem,R,times", [
    (750, 9, {16: 21.7, 8: 37.8, 4: 52.3, 2: 81.2, 1: 142.4}),
    (3072, 9, {4: 52.2, 8: 58.6, 16: 60.4, 2: 83.0, 1: 142.6}),
    (3072, 24, {8: 84.9, 4: 97.3, 16: 107.9, 32: 114.0, 2: 188.0, 1: 368.2}),
    (7986, 5, {2: 56.3, 4: 66.4, 8: 77.1, 1: 82.8}),
    (7986, 16, {4: 123.6, 16: 132.8, 2: 138.3, 8: 142.4, 1: 249.2}),
    (16464, 3, {1: 56.2, 2: 66.3, 4: 77.1}),
    (16464, 16, {2: 238.1, 8: 244.8, 16: 261.0, 4: 269.2, 1: 275.2}),
    (31104, 9, {1: 267.1, 2: 332.7, 4: 354.9, 8: 448.4, 16: 481.2}),
    (73728, 2, {1: 140.9, 2: 149.0}),
    (73728, 30, {1: 1933.2, 2: 1936.1, 8: 2049.7, 4: 2077.6, 16: 2093.6, 32: 2249.7}),
    (82944, 16, {2: 1173.1, 4: 1177.9, 8: 1198.8, 16: 1265.4, 1: 1298.0}),
    (146124, 16, {4: 2030.4, 2: 2037.4, 1: 2067.5, 8: 2084.6, 16: 2216.8}),
    (1029000, 16, {1: 13620.4, 2: 13726.2, 4: 13958.7, 8: 14459.7, 16: 15506.9})])
def test_lanes_of_the_sensitivities(rules, n_elem, R, times):
    assert near_best(rules.f64_adjoint_split(ctypes.c_long(n_elem), R, SMS), times)
