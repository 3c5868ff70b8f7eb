"""The tuner's search (csrc/tune_search.h, compiled here for the host) with made-up times: it starts
from the shape a level runs untuned and never ends on a slower one."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1703_10435_gb300", "csrc")
CUDA = "/usr/local/cuda/include"
SHIM = r'''
#include "tune_search.h"
typedef double (*cost_t)(int, int, int, int, int, int);
extern "C" void search(int degree, int N, int n_I, cost_t cost, int* first, int* out, double* ms) {
    int n = 0;
    const mhm::Tuning t = mhm::tune_descend(mhm::untuned(degree, N, n_I), ms, [&](const mhm::Tuning& s, double* v) {
        *v = cost(s.chunk, s.blocks_per_sm, s.nbuf, s.l2pf, s.pf_all, s.op_policy);
        if (n++ == 0) first[0] = s.chunk, first[1] = s.blocks_per_sm, first[2] = s.nbuf;
        return true;
    });
    out[0] = t.chunk, out[1] = t.blocks_per_sm, out[2] = t.nbuf;
}
'''
COST = ctypes.CFUNCTYPE(ctypes.c_double, *[ctypes.c_int] * 6)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++") or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no g++ or CUDA headers")
    d = tmp_path_factory.mktemp("tune")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "libtune.so")
    subprocess.check_call(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                           "-I", CUDA, "-o", so, str(d / "shim.cpp")])
    return ctypes.CDLL(so)


@pytest.mark.parametrize("degree,N,n_I,blocks", [(1, 8, 18, 4), (1, 16, 18, 4), (1, 32, 6, 4), (1, 32, 18, 3)])
def test_starts_from_the_untuned_shape(lib, degree, N, n_I, blocks):
    def cost(chunk, bps, nbuf, l2pf, pf_all, policy):
        """The untuned shape is the best; beside it a valley with a deeper ring."""
        if (bps, nbuf) == (blocks, 2):
            return 1.0 + 0.01 * (l2pf > 0) + 0.01 * pf_all + 0.01 * (policy != 1) + 0.01 * (chunk != 8192)
        return 1.1 if nbuf == 4 and bps == 7 - blocks else 1.2 - 0.01 * nbuf
    first, out, ms = (ctypes.c_int * 3)(), (ctypes.c_int * 3)(), ctypes.c_double()
    lib.search(degree, N, n_I, COST(cost), first, out, ctypes.byref(ms))
    assert list(first) == [8192, blocks, 2]
    assert list(out) == [8192, blocks, 2] and ms.value == 1.0
