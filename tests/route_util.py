"""The choice of a round's kernels (``csrc/dq_route.h``), compiled for the host."""
import ctypes as C
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2107_14575_b200", "csrc")
WARPS, CTAS, TWO = 0, 1, 2               # RoundRoute
B200_SMS = 148


def compile_route(directory):
    """``route(groups, buckets, bucket, M, sms)``: the kernels a round of ``groups`` 32-element groups per worker in
    ``buckets`` buckets of ``bucket`` elements (0: whole tensors) takes; ``linf``: l-infinity norms; ``lost``: under the test hook of the waits."""
    src, lib = os.path.join(str(directory), "route.cpp"), os.path.join(str(directory), "route.so")
    with open(src, "w") as fh:
        fh.write('#include "dq_route.h"\nextern "C" int route(int64_t positions, int64_t warps, int gpb, int M, int given, int linf, int lost) '
                 '{ return dq_route_of(positions, warps, gpb, M, given != 0, linf != 0, lost != 0); }\n')
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-I", CSRC, src, "-o", lib], check=True)
    f = C.CDLL(lib).route
    f.argtypes = [C.c_int64, C.c_int64] + [C.c_int] * 5

    def route(groups, buckets, bucket, M, sms=B200_SMS, lost=False, linf=False):
        gpb = bucket // 32 if bucket else 1 << 20
        given = bucket == 0 or (gpb & (gpb - 1) != 0 and gpb > 31)
        if given:
            positions = -(-groups // 32)
        else:
            positions = buckets if gpb > 32 else -(-buckets // (32 // gpb))
        return f(positions, sms * 4 * 4, gpb, M, given, linf, lost)
    return route
