"""Which plans run their forward dynamics with three lanes per request
(csrc/fleet_rule.h, compiled for the host): the form that was measured faster by a
tenth or more on GB300 (152 SMs), over chain lengths and request counts on both sides
of the line, and the list schedule itself."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1609_04493_gb300", "csrc")

SRC = r"""
#include "fleet_rule.h"
extern "C" int takes_lanes(const int *n, int fd, int id, int ext_groups, int sms)
{
    return rd_fleet_takes_lanes(std::vector<int>(n, n + fd), std::vector<int>(n + fd, n + fd + id),
                                ext_groups, 10, sms);
}
extern "C" double schedule(const double *t, int count, int workers)
{
    return rd_list_schedule(std::vector<double>(t, t + count), workers);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("rule")
    src, so = str(d / "r.cpp"), str(d / "r.so")
    with open(src, "w") as fh:
        fh.write(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.schedule.restype = ctypes.c_double
    return lib


def takes_lanes(rule, fd, inverse=(), sms=152):
    fd, inverse = (np.sort(np.asarray(n, dtype=np.int32))[::-1] for n in (fd, inverse))
    ext = int(np.sum(fd[::32] > 64))
    n = np.concatenate([fd, inverse])
    return bool(rule.takes_lanes(n.ctypes.data_as(ctypes.POINTER(ctypes.c_int)), len(fd), len(inverse), ext, sms))


# lengths, forward-dynamics requests, us with one thread and with three lanes per request
MEASURED = [
    (1, 2, 4000, 12.5, 10.3), (1, 2, 12000, 13.0, 10.9), (1, 2, 30000, 13.8, 18.3), (1, 2, 120000, 22.6, 47.1),
    (3, 5, 12000, 26.5, 18.6), (3, 5, 30000, 26.7, 35.1), (3, 5, 120000, 67.0, 110.8),
    (7, 7, 1, 32.0, 18.5), (7, 7, 4000, 36.4, 22.7), (7, 7, 12000, 38.1, 26.7), (7, 7, 18240, 39.0, 43.2),
    (7, 7, 30000, 40.7, 61.5), (7, 7, 120000, 124.2, 194.5),
    (6, 12, 12000, 57.7, 33.3), (6, 12, 18240, 59.2, 47.2), (6, 12, 30000, 59.7, 72.9),
    (6, 30, 18240, 143.4, 88.4), (6, 30, 60000, 184.3, 258.6),
    (32, 32, 12000, 166.4, 96.1), (32, 32, 30000, 182.3, 270.3),
    (60, 64, 12000, 330.8, 191.8), (60, 64, 30000, 371.9, 535.5),
    (6, 100, 4000, 855.6, 293.9), (6, 100, 30000, 1110.1, 536.9), (6, 100, 60000, 1415.0, 1067.1),
    (65, 65, 10000, 570.0, 287.2), (65, 65, 13000, 585.2, 460.3), (65, 65, 20000, 608.4, 545.4),
    (100, 128, 12000, 1160.3, 603.2), (100, 128, 18240, 1158.5, 973.7), (100, 128, 30000, 1215.5, 1556.7),
]
# the same with one forward-dynamics request in `every`, `count` requests in all
MIXED = [
    (3, 5, 5, 60000, 27.4, 20.5), (3, 5, 5, 120000, 31.4, 34.9), (3, 5, 5, 250000, 47.2, 68.0),
    (7, 7, 20, 120000, 38.8, 29.8), (7, 7, 20, 250000, 46.7, 56.6), (7, 7, 5, 30000, 38.5, 28.9),
    (7, 7, 5, 120000, 41.3, 57.4), (7, 7, 5, 250000, 78.4, 107.9), (7, 7, 2, 60000, 41.4, 61.6),
    (6, 30, 5, 60000, 140.4, 83.9), (6, 30, 5, 250000, 229.2, 306.1),
    (32, 32, 5, 30000, 171.0, 123.9), (32, 32, 5, 120000, 201.9, 348.2), (32, 32, 2, 30000, 172.3, 192.6),
    (60, 64, 5, 60000, 352.9, 286.6), (6, 100, 5, 20000, 944.0, 366.0), (6, 100, 5, 120000, 1057.4, 591.1),
]


@pytest.mark.parametrize("lo,hi,count,one,three", MEASURED)
def test_the_faster_form_is_taken(rule, lo, hi, count, one, three):
    for seed in range(3):
        n = np.random.default_rng(seed).integers(lo, hi + 1, count)
        assert takes_lanes(rule, n) == (three < one)


@pytest.mark.parametrize("lo,hi,every,count,one,three", MIXED)
def test_the_faster_form_is_taken_beside_inverse_dynamics(rule, lo, hi, every, count, one, three):
    n = np.random.default_rng(7).integers(lo, hi + 1, count)
    assert takes_lanes(rule, n[:count // every], n[count // every:]) == (three < one)


@pytest.mark.parametrize("lo,hi,count,one,three", [(1, 2, 4000, 6.4, 8.1), (1, 2, 60000, 10.3, 8.3),
                                                   (3, 5, 9000, 8.6, 10.1), (3, 5, 120000, 21.5, 16.6),
                                                   (7, 7, 60000, 17.7, 20.7), (6, 30, 60000, 31.1, 48.5),
                                                   (32, 32, 30000, 46.4, 64.5), (100, 128, 38000, 136.1, 231.9)])
def test_without_forward_dynamics(rule, lo, hi, count, one, three):
    assert takes_lanes(rule, [], np.random.default_rng(2).integers(lo, hi + 1, count)) == (three < one)


def test_the_line_moves_with_the_gpu(rule):
    n = np.full(6080, 7)  # ten of each of 8 x 76 units
    assert not takes_lanes(rule, []) and takes_lanes(rule, n, sms=76) and not takes_lanes(rule, np.full(12160, 7), sms=76)


def test_list_schedule(rule):
    t = np.random.default_rng(1).uniform(1, 9, 200)
    for workers in (1, 3, 50, 400):
        free = [0.0] * workers
        for x in t:
            k = int(np.argmin(free))
            free[k] += x
        got = rule.schedule(t.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), len(t), workers)
        assert abs(got - max(free)) < 1e-9
