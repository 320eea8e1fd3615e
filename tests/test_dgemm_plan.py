"""Tile and K split of the FP64 GEMM (csrc/dgemm_plan.h), compiled for the host: every plan
covers K with non-empty ranges, fits the grid and its workspace -- from an empty K to the
largest one, where the arithmetic has to be 64-bit."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_13184_gb300", "csrc")


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("dgemm_plan")
    (d / "p.cpp").write_text('#include "dgemm_plan.h"\n'
                             'extern "C" void plan(int M, int N, int K, size_t ws, int* o) {\n'
                             '    const ctm::GemmPlan p = ctm::dgemm_plan(M, N, K, ws);\n'
                             '    o[0] = p.tm; o[1] = p.tn; o[2] = p.splits; o[3] = p.kchunk;\n}\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "p.so"), str(d / "p.cpp")],
                   check=True)
    f = ctypes.CDLL(str(d / "p.so")).plan
    f.argtypes = [ctypes.c_int] * 3 + [ctypes.c_size_t, ctypes.POINTER(ctypes.c_int)]

    def call(M, N, K, ws):
        o = (ctypes.c_int * 4)()
        f(M, N, K, ws, o)
        return tuple(o)
    return call


MAX = 2**31 - 1


@pytest.mark.parametrize("K", [0, 1, 15, 16, 17, 300, 70000, 2**30, 2**30 + 1, 1200000000, MAX - 16, MAX])
@pytest.mark.parametrize("M,N", [(1, 1), (9, 1), (144, 144), (33, 73), (5000, 36), (1, 4194240), (20000, 40)])
def test_plan_covers_k(plan, M, N, K):
    for ws in (0, 1 << 24):
        tm, tn, splits, kchunk = plan(M, N, K, ws)
        assert tm in (1, 2, 4) and 1 <= tn <= 9
        assert -(-N // (8 * tn)) <= 65535
        assert 1 <= splits <= 256
        if splits > 1:
            assert splits * M * N <= ws
            assert kchunk > 0 and (splits - 1) * kchunk < K <= splits * kchunk
