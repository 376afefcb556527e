"""The choice between one kernel and two for a round (``csrc/dq_route.h``), compiled for the host, against the measured
times that are quoted beside it: it takes the faster side of every line, or one within 3 % of it."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_14575_b200", "csrc")

# bucket (0: whole tensors), elements, M, us in one pass, us by two kernels
LINES = [(512, 20001, 4, 10.9, 11.9), (512, 20001, 32, 58, 15), (512, 70001, 4, 13.5, 13.2), (512, 600001, 4, 10.6, 12.8),
         (512, 600001, 8, 17.3, 15.1), (512, 600001, 32, 58, 30), (512, 1500001, 8, 22.0, 21.8), (512, 1500001, 32, 73, 56),
         (512, 3000001, 8, 31.5, 34.4), (512, 3000001, 32, 109, 102), (512, 4200001, 32, 129, 136), (512, 10000001, 32, 263, 308),
         (2048, 600001, 4, 12.2, 13.8), (2048, 600001, 8, 19.9, 16.9), (2048, 1500001, 32, 82, 63), (2048, 5200001, 32, 179, 189),
         (480, 600001, 8, 25.7, 18.7), (480, 1500001, 4, 13.7, 19.9), (480, 3000001, 8, 45, 41), (480, 8000001, 8, 85, 94),
         (96, 20001, 4, 19.4, 16.1), (96, 600001, 8, 32, 21), (96, 1500001, 4, 21.6, 24.8), (96, 3000001, 8, 62, 49),
         (0, 600001, 32, 53, 42), (0, 3000001, 8, 42, 49)]


class Query(C.Structure):
    _fields_ = [("positions", C.c_int64), ("units", C.c_int64), ("M", C.c_int32), ("given", C.c_int32), ("odd_buckets", C.c_int32)]


@pytest.fixture(scope="module")
def one_pass(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    src, lib = str(d / "route.cpp"), str(d / "route.so")
    with open(src, "w") as fh:
        fh.write('#include "dq_route.h"\nextern "C" int one_pass(RouteQuery q) { return dq_one_pass(q); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-I", CSRC, src, "-o", lib], check=True)
    f = C.CDLL(lib).one_pass
    f.argtypes = [Query]
    return lambda *a: bool(f(Query(*a)))


def _query(bucket, d, M):
    groups, units = -(-d // 32), 148 * 4 * 4
    if bucket == 0:
        return -(-groups // 32), units, M, 1, 0
    gpb, nb = bucket // 32, -(-d // bucket)
    if gpb > 32:
        return nb, units // (gpb // 32), M, 0, 0
    return -(-nb // (32 // gpb)), units, M, 0, 32 // gpb if gpb & (gpb - 1) else 0


@pytest.mark.parametrize("bucket,d,M,one,two", LINES)
def test_the_faster_side_of_every_measured_line(one_pass, bucket, d, M, one, two):
    taken = one if one_pass(*_query(bucket, d, M)) else two
    assert taken <= 1.03 * min(one, two)


def test_one_worker_and_whole_turns_take_one_pass(one_pass):
    assert one_pass(69, 2368, 1, 0, 0) and one_pass(2 * 2368, 2368, 32, 0, 10)
