"""The panel plan of the doubled adjoint (csrc/adjoint_plan.cuh), compiled for the host: what is asked for when an
allocation fails."""
import ctypes
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_05264_gb300", "csrc")


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cpp", d / "libplan.so"
    # bytes of the plan and of every smaller one, until there is none
    src.write_text('#include "adjoint_plan.cuh"\nusing namespace tbk;\n'
                   'extern "C" int sizes(int npan, int windowed, int batch, int defer, long prefix, long* out, int* wait) {\n'
                   "  AdjointPlan p;\n  p.npan = p.seg = npan;\n  p.panel = 1000;\n  p.windowed = windowed;\n"
                   "  p.batch = batch;\n  p.defer = defer;\n  p.prefix_tail = prefix;\n"
                   "  int n = 0;\n  do { out[n] = p.bytes(); wait[n++] = p.defer; } while (n < 8 && p.shrink());\n"
                   "  return n;\n}\n")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).sizes
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_long, ctypes.c_void_p, ctypes.c_void_p]

    def call(npan, windowed=0, batch=0, defer=0, prefix=0):
        out, wait = (ctypes.c_long * 8)(), (ctypes.c_int * 8)()
        n = f(npan, windowed, batch, defer, prefix, out, wait)
        return list(out[:n]), list(wait[:n])
    return call


def _segments(npan, ybar, probe=0):
    seg = 4 * math.ceil(max(2, math.ceil(math.sqrt(2 * npan))) / 4)
    nseg = math.ceil(npan / seg)
    return 1000 * (seg + 1 + (2 * nseg if nseg > 1 else 0) + 1 + ybar + probe)


@pytest.mark.parametrize("npan", [1, 2, 3, 4, 9, 18, 63, 315, 1238])
@pytest.mark.parametrize("defer", [0, 1, 2, 9, 64])
def test_plans_shrink_to_two_ybar_panels_and_then_to_segments(sizes, npan, defer):
    got, wait = sizes(npan, defer=min(defer, npan))
    d = min(defer, npan)
    want = [1000 * (npan + 2 + (d + 1 if d > 1 else 2))]
    if d > 1:
        want.append(1000 * (npan + 4))
    if npan > 2 and _segments(npan, 2) < 1000 * (npan + 4):
        want.append(_segments(npan, 2))
        assert wait[-1] == 0
    assert got == want
    assert all(a > b for a, b in zip(got, got[1:]))


def test_windows_and_batches_keep_their_panels(sizes):
    assert sizes(63, windowed=1)[0] == [1000 * (63 + 2 + 6), _segments(63, 6)]
    assert sizes(63, windowed=1, batch=1, prefix=40000)[0] == [47000, _segments(63, 6, 1)]
    assert sizes(63, batch=1, prefix=40000)[0] == [43000, _segments(63, 2, 1)]
