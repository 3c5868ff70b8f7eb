"""The largest bordered matrices of the 2-D frontal elimination (M = 178 and 180 rows: 49 loads,
sixteen warps with their last block rows in use) and the 3-D refinement kernel on a full-size mesh."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import tet3d as T
from oracle.local import solve_local
from oracle.mesh import build_mesh
from oracle.run import source_fn
from paper_1703_10435_gb300 import mhm, workloads as W
from tests._blocks import assert_blocks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10435_gb300 import build
    build.build()


@pytest.mark.parametrize("P,r,m,l", [(1, 7, 16, 0), (2, 6, 16, 0), (1, 6, 16, 0)])
def test_blocks_vs_oracle_with_49_loads(P, r, m, l):
    from paper_1703_10435_gb300.pipeline import Pipeline
    w = W.Workload("t", 1, 1, r, P, m, l, "log_uniform", "sinsin", 1.0, 1.0, seed=3)
    kap = W.kappa_for(w) ** 0.25   # contrast 10
    p = Pipeline.for_workload(w, 0, mhm.MHM_FP64)
    p.local(torch.as_tensor(kap, device="cuda"), mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 1.0))
    torch.cuda.synchronize()
    assert int(p.status.abs().sum()) == 0 and p.iters.cpu().tolist() == [1, 1]
    AK, EK, BK, FK = p.blocks()
    mesh = build_mesh(1, 1, m, l)
    n = (P * 2 ** r + 1) * (P * 2 ** r + 2) // 2
    # 10 u cond; the P1 / P2 stiffness on n points has cond of about 12 n times the contrast
    tol = max(1e-10, 10 * 1.1e-16 * 12 * n * 10)
    for K in range(2):
        assert_blocks(AK[K], EK[K], BK[K], FK[K], solve_local(mesh, K, r, P, kap[K], source_fn("sinsin", 1.0, 1.0)), tol, K)


def test_3d_refinement_full_size():
    """12288 tetrahedra, P2 r = 2, m = 4 with the FP64 re-solve turned off, so that the refinement
    kernel gives every block: converged in two passes or more, sampled elements against the oracle
    and all of them against the FP64 elimination on the Gram scale."""
    nc, r, P, m = 8, 2, 2, 4
    M = mhm.Mesh3D(nc, r, P, m)
    o = T.build_mesh3d(nc, m)
    rng = np.random.default_rng(2026)
    kappa = 10.0 ** rng.uniform(-1, 1, (M.n_K, 64))
    kd = torch.as_tensor(kappa, device="cuda")
    src, f = mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0), T.source3d_fn("sinsinsin", 1.0, 2.0)

    def run(precision, opts=None):
        f64 = dict(dtype=torch.float64, device="cuda")
        b = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
             torch.zeros(M.n_K, **f64), torch.full((M.n_K,), -7, dtype=torch.int32, device="cuda"),
             torch.full((M.n_K,), -9, dtype=torch.int32, device="cuda")]
        mhm.mhm3d_local_solve_batch(M, kd, src, *b[:5], precision=precision, opts=opts, iters=b[5])
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x in b]
    mx, ref = run(mhm.MHM_MIXED, mhm.Opts3D(8, 1e-9, 1)), run(mhm.MHM_FP64)
    assert np.all(mx[4] == 0) and mx[5].min() >= 2 and mx[5].max() <= 8
    assert np.all(ref[4] == 0) and np.all(ref[5] == 1)
    amp = 12.0 * math.pi ** 2 / M.n_K
    for K in [0, M.n_K - 1] + [int(k) for k in rng.choice(M.n_K, 4, replace=False)]:
        loc = T.solve_local3d(o, K, r, P, kappa[K], f)
        d = np.sqrt(np.abs(np.diag(loc.AK)))
        assert (np.abs(mx[0][K] - loc.AK) / np.outer(d, d)).max() < 1e-10
        scale = max(np.abs(loc.EK).max(), np.abs(loc.AK).max() * abs(loc.FK) / np.abs(loc.BK).max())
        assert np.abs(mx[1][K] - loc.EK).max() < 1e-10 * scale
        assert np.abs(mx[2][K] - loc.BK).max() < 1e-10 * np.abs(loc.BK).max()
        assert abs(mx[3][K] - loc.FK) < 1e-13 * amp
    # the target of 1e-9 per column, squared by the corrected form, and the FP64 elimination's rounding
    d = np.sqrt(np.abs(np.einsum("kii->ki", ref[0])))
    assert float((np.abs(mx[0] - ref[0]) / (d[:, :, None] * d[:, None, :])).max()) < 1e-10
    assert np.abs(mx[1] - ref[1]).max() <= 1e-10 * np.abs(ref[1]).max()
    assert np.array_equal(mx[2], ref[2]) and np.array_equal(mx[3], ref[3])
