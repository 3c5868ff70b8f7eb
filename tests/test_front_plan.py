"""Step tables of the 2-D frontal elimination (csrc/front_plan.cpp, compiled here for the host): run
step by step on random element matrices they eliminate the assembled matrix, with every node in
a slot of its own; orders whose front is too large are refused without building their schedule."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_10435_gb300", "csrc")
SHIM = r'''
#include <algorithm>
#include <chrono>
#include "front_plan.h"
static mhm::FrontPlan plan;
extern "C" double make_plan(int P, int N, int* info) {
    const auto t = std::chrono::steady_clock::now();
    plan = mhm::front_plan_2d(P, N);
    const double s = std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count();
    info[0] = plan.steps, info[1] = plan.slots, info[2] = plan.ncp, info[3] = (int)plan.tab.size();
    return s;
}
extern "C" void get_plan(unsigned* out) { std::copy(plan.tab.begin(), plan.tab.end(), out); }
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "libplan.so")
    subprocess.check_call(["g++", "-O2", "-shared", "-fPIC", "-std=c++17", "-I", CSRC, "-o", so, str(d / "shim.cpp"),
                           os.path.join(CSRC, "front_plan.cpp")])
    L = ctypes.CDLL(so)
    L.make_plan.restype = ctypes.c_double
    return L


def _plan(L, P, N):
    info = (ctypes.c_int * 4)()
    seconds = L.make_plan(P, N, info)
    tab = np.zeros(max(info[3], 1), np.uint32)
    L.get_plan(tab.ctypes.data_as(ctypes.c_void_p))
    steps, slots, ncp = info[0], info[1], info[2]
    return steps, slots, tab[:4 * steps].reshape(-1, 4), tab[4 * steps:info[3]].reshape(steps, ncp, 2) if steps else None, seconds


def _triangles(P, N):
    """Nodes (lattice points) of the fine triangles in kappa order, and whether they point up."""
    for j in range(N):
        for up in (1, 0):
            for i in range(N - j if up else N - 1 - j):
                v = [(i, j), (i + 1, j), (i, j + 1)] if up else [(i + 1, j), (i + 1, j + 1), (i, j + 1)]
                pts = [(P * x, P * y) for x, y in v]
                if P == 2:
                    pts += [(a[0] + b[0], a[1] + b[1]) for a, b in ((v[1], v[2]), (v[2], v[0]), (v[0], v[1]))]
                yield pts, up


@pytest.mark.parametrize("P,r", [(1, 0), (1, 1), (1, 2), (1, 3), (1, 4), (2, 0), (2, 1), (2, 2), (2, 3)])
def test_tables_eliminate_the_assembled_matrix(lib, P, r):
    N = 2 ** r
    steps, slots, ev, cp, _ = _plan(lib, P, N)
    assert slots == (N + 1 if P == 1 else 2 * N + 3)
    rng = np.random.default_rng(10 * P + r)
    nb = 3 if P == 1 else 6
    Ke = [(lambda B: B @ B.T + nb * np.eye(nb))(rng.standard_normal((nb, nb))) for _ in range(2)]   # up, down
    kap = rng.uniform(0.5, 2.0, N * N)
    nodes = {}
    tris = list(_triangles(P, N))
    for pts, _ in tris:
        for p in pts:
            nodes.setdefault(p, len(nodes))
    n, R = len(nodes), 3
    A = np.zeros((n, n))
    mass = np.zeros(n, int)
    for (pts, up), k in zip(tris, kap):
        ix = [nodes[p] for p in pts]
        A[np.ix_(ix, ix)] += k * Ke[0 if up else 1]
        for a, i in enumerate(ix):
            mass[i] += P == 1 or a >= 3
    G = rng.standard_normal((n, R))
    F = np.zeros((R + slots, R + slots))
    held = [None] * slots
    flat = np.zeros(72)
    for d in range(2):
        flat[36 * d:36 * d + nb * nb] = Ke[d].ravel()
    entered = []
    for (e0, pt, info, piv), rows in zip(ev, cp):
        ps, zs, m = int(e0) & 255, int(e0) >> 8 & 255, int(e0) >> 16
        assert all(h is None for h in held[m:])
        w, wnew, row = None, 0.0, np.zeros(R + slots)
        if ps != 255:
            assert held[ps] == (int(piv) & 0xffff, int(piv) >> 16)
            w = F[R + ps].copy()
            F[R + ps] = F[:, R + ps] = 0.0
            held[ps] = None
        if zs != 255:
            p = (int(pt) & 0xffff, int(pt) >> 16)
            i = nodes[p]
            entered.append(p)
            assert held[zs] is None and zs < m
            held[zs] = p
            assert int(info) & 255 == mass[i]
            assert int(info) >> 8 == ((p[0] + p[1] == P * N) | (p[0] == 0) << 1 | (p[1] == 0) << 2)
            diag = 0.0
            for x, y in rows:
                sl, t0, t1 = int(x) & 255, int(y) & 0xffff, int(y) >> 16
                v = 0.0 if t0 == 0xffff else kap[t0] * flat[int(x) >> 8 & 255]
                v += 0.0 if t1 == 0xffff else kap[t1] * flat[int(x) >> 16 & 255]
                if sl == 253:
                    diag += v
                elif sl == 254:
                    wnew = v
                elif sl != 255:
                    row[R + sl] = v
            row[:R] = G[i]
            row[R + zs] = diag
            F[R + zs], F[:, R + zs] = row, row
        if w is not None:
            d = w[R + ps]
            w[R + ps] = 0.0
            if zs != 255:
                w[R + zs] = wnew
            F -= np.outer(w, w) / d
    assert sorted(entered) == sorted(nodes)
    want = -G.T @ np.linalg.solve(A, G)
    assert np.abs(F[:R, :R] - want).max() < 1e-12 * np.abs(want).max()   # (cond A about 1e2)


def test_too_large_fronts_are_refused_at_once(lib):
    """P2 r = 7 (259 slots): less time than the schedule of P2 r = 5 takes."""
    assert _plan(lib, 2, 128)[0] == 0
    refused = min(_plan(lib, 2, 128)[4] for _ in range(3))
    assert refused < min(_plan(lib, 2, 32)[4] for _ in range(3))
    steps, slots = _plan(lib, 2, 64)[:2]
    assert (steps, slots) == (8516, 131)
    steps, slots = _plan(lib, 1, 128)[:2]
    assert (steps, slots) == (8514, 129)
