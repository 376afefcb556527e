"""Which of its kernels a round takes (``dq_round_route`` of ``csrc/dq_route.h``, compiled for the host), against measured times
of the three: the one taken is within 16 % of the fastest on every line (the worst of the fit)."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_14575_b200", "csrc")

# bucket (0: whole tensors), elements, M, us by warps, by CTAs, by two kernels
LINES = [(512, 16013, 4, 10, 6, 12), (512, 16013, 16, 27, 11, 13), (512, 16013, 32, 49, 17, 15), (512, 456263, 4, 11, 7, 13),
         (512, 456263, 16, 28, 14, 20), (512, 797387, 8, 18, 13, 18), (512, 1393555, 16, 36, 30, 32), (512, 2435449, 16, 54, 42, 48),
         (512, 7438555, 8, 57, 64, 71), (2048, 16013, 4, 11, 8, 12), (2048, 16013, 16, 30, 20, 16), (2048, 456263, 8, 17, 14, 18),
         (2048, 1393555, 8, 23, 21, 29), (2048, 3050001, 16, 60, 68, 67), (96, 16013, 4, 15, 7, 15), (96, 456263, 8, 24, 12, 19),
         (96, 4256315, 8, 60, 58, 66), (0, 16013, 4, 13, 10, 16), (0, 456263, 8, 20, 14, 21), (0, 2435449, 8, 47, 44, 47)]


class Query(C.Structure):
    _fields_ = [("positions", C.c_int64), ("units", C.c_int64), ("M", C.c_int32), ("given", C.c_int32), ("odd_buckets", C.c_int32)]


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    src, lib = str(d / "route.cpp"), str(d / "route.so")
    with open(src, "w") as fh:
        fh.write('#include "dq_route.h"\nextern "C" int route(RouteQuery q, int tiles, int pairs) '
                 '{ return dq_round_route(q, tiles != 0, pairs != 0); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-I", CSRC, src, "-o", lib], check=True)
    f = C.CDLL(lib).route
    f.argtypes = [Query, C.c_int, C.c_int]
    return f


def _query(bucket, d, M):
    groups, units = -(-d // 32), 148 * 4 * 4
    if bucket == 0:
        return Query(-(-groups // 32), units, M, 1, 0)
    gpb, nb = bucket // 32, -(-d // bucket)
    if gpb > 32:
        return Query(nb, units // (gpb // 32), M, 0, 0)
    return Query(-(-nb // (32 // gpb)), units, M, 0, 32 // gpb if gpb & (gpb - 1) else 0)


@pytest.mark.parametrize("bucket,d,M,warps,ctas,two", LINES)
def test_close_to_the_fastest_of_every_measured_line(route, bucket, d, M, warps, ctas, two):
    taken = (warps, ctas, two)[route(_query(bucket, d, M), 1, bucket == 2048)]
    assert taken <= 1.16 * min(warps, ctas, two)


def test_buckets_of_4096_never_take_the_kernel_they_have_no_form_of(route):
    for d in (1, 70001, 1 << 20, 1 << 24):
        for M in (1, 2, 8, 32):
            assert route(_query(4096, d, M), 0, 0) != 1


def test_which_buckets_a_cta_has_a_form_for(tmp_path):
    """Teams are pairs of warps there: buckets of 4096 go by warps or by two kernels whatever their size, the others, given
    norms of any bucket among them, by CTAs where they are small."""
    import route_util
    route = route_util.compile_route(tmp_path)
    for d in (1, 70001, 1 << 20, 1 << 24):
        groups = -(-d // 32)
        for M in (1, 2, 8, 32):
            assert route(groups, -(-d // 4096), 4096, M) != route_util.CTAS
    for bucket in (32, 64, 96, 480, 512, 992, 1024, 2048, 1056, 4064, 0):
        nb = -(-70001 // bucket) if bucket else 1
        assert route(-(-70001 // 32), nb, bucket, 4) == route_util.CTAS


@pytest.mark.parametrize("bucket", [32, 96, 480, 512, 1024, 2048, 4096, 1056, 0])
def test_under_the_hook_of_the_waits_a_round_takes_kernels_that_have_one_to_lose(tmp_path, bucket):
    """... the ones the same size would take if there were no kernel by CTAs."""
    import route_util
    route = route_util.compile_route(tmp_path)
    for d in (1, 3001, 70001, 600001, 1 << 20, 3300001, 1 << 24):
        groups, nb = -(-d // 32), -(-d // bucket) if bucket else 1
        for M in (1, 2, 3, 8, 40):
            lost = route(groups, nb, bucket, M, lost=True)
            assert lost != route_util.CTAS
            if route(groups, nb, bucket, M) == route_util.WARPS and bucket != 2048:
                assert lost == route_util.WARPS
