"""The 3-D step (local solves with the sin sin sin source, skeleton gather) takes no device memory
of its own: nothing from the stream-ordered pool, and a graph of it replays on new inputs with the
bits of the call."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_10435_gb300 import mhm

pytestmark = pytest.mark.gpu

POOL_USED_MEM_HIGH = 8   # CU_MEMPOOL_ATTR_USED_MEM_HIGH


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10435_gb300 import build
    build.build()


def _pool():
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    dev, pool = ctypes.c_int(0), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    return cu, pool


@pytest.mark.parametrize("precision", [mhm.MHM_FP64, mhm.MHM_MIXED])
@pytest.mark.parametrize("nc,r,P,m", [(1, 0, 2, 1), (1, 1, 1, 1), (3, 1, 2, 4), (1, 2, 2, 4), (2, 2, 2, 16)])
def test_step_allocates_nothing_and_replays(nc, r, P, m, precision):
    M = mhm.Mesh3D(nc, r, P, m)
    f64 = dict(dtype=torch.float64, device="cuda")
    o = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
         torch.zeros(M.n_K, **f64), torch.zeros(M.n_K, dtype=torch.int32, device="cuda"),
         torch.zeros(M.nnz, **f64), torch.zeros(M.n_lambda, **f64)]
    src = mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0)
    rng = np.random.default_rng(11)
    kaps = [torch.as_tensor(10.0 ** rng.uniform(-1, 1, (M.n_K, 8 ** r)), device="cuda") for _ in range(2)]
    kap = kaps[0].clone()

    def step(stream=None):
        mhm.mhm3d_local_solve_batch(M, kap, src, *o[:5], precision=precision, stream=stream)
        mhm.mhm3d_assemble_skeleton(M, o[0], o[1], o[5], o[6], stream)
    step()
    torch.cuda.synchronize()
    cu, pool = _pool()
    high = ctypes.c_uint64(0)
    assert cu.cuMemPoolSetAttribute(pool, POOL_USED_MEM_HIGH, ctypes.byref(high)) == 0
    step()
    torch.cuda.synchronize()
    assert cu.cuMemPoolGetAttribute(pool, POOL_USED_MEM_HIGH, ctypes.byref(high)) == 0
    assert high.value == 0
    want = []
    for k in kaps:
        kap.copy_(k)
        step()
        torch.cuda.synchronize()
        assert int(o[4].abs().sum()) == 0
        want.append([x.clone() for x in o])
    graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=s):
        step(s)
    for k, w in zip(kaps, want):
        kap.copy_(k)
        for x in o:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(o, w))


@pytest.mark.parametrize("precision", [mhm.MHM_FP64, mhm.MHM_MIXED])
def test_ranges_of_elements_match_the_full_call(precision):
    """Ranges that start and end inside a group of 24 (the kernels order a range by type)."""
    M = mhm.Mesh3D(2, 1, 2, 4)
    kap = torch.as_tensor(10.0 ** np.random.default_rng(5).uniform(-1, 1, (M.n_K, 8)), device="cuda")
    src = mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0)
    f64 = dict(dtype=torch.float64, device="cuda")

    def run(ranges):
        o = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
             torch.zeros(M.n_K, **f64), torch.full((M.n_K,), -7, dtype=torch.int32, device="cuda")]
        for K0, K1 in ranges:
            mhm.mhm3d_local_solve_batch(M, kap, src, *o, K0=K0, K1=K1, precision=precision)
        return o
    full = run([(0, 0)])
    assert int(full[4].abs().sum()) == 0
    cuts = [0, 1, 24, 31, 55, 56, 101, 149, 192]
    assert all(torch.equal(a, b) for a, b in zip(full, run(list(zip(cuts, cuts[1:])))))
    part = run([(7, 61)])
    assert all(torch.equal(a[7:61], b[7:61]) for a, b in zip(full, part))
    assert bool((part[4][:7] == -7).all()) and bool((part[4][61:] == -7).all())
