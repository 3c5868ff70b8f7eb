"""The FP64 frontal elimination at the sizes where its layout changes: the bordered matrix has
M = R + slots rows (R = 3 m (l + 1) + 1 loads; P1: 2^r + 1 slots, P2: 2 2^r + 3), handled in
4-row tiles by one warp up to M = 64 and by 4, 8 or 16 warps above, and by a window in global
memory beyond (P2 r = 7).  Both elements of a one-square mesh, sin sin source (its loads by
the addition theorem), against the oracle entry by entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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


# (P, r, m, l): M and the warps that share it
CASES = [(1, 0, 1, 0),    # 7, one warp, 4 rows of tiles
         (1, 3, 2, 0),    # 16: the last size of 4 rows of tiles
         (1, 3, 3, 0),    # 19
         (1, 4, 2, 1),    # 30, not a multiple of 4
         (1, 5, 2, 0),    # 40: the last of 10
         (2, 4, 1, 1),    # 42
         (1, 5, 3, 1),    # 52: the last of 13
         (1, 5, 7, 0),    # 55
         (1, 5, 10, 0),   # 64: the last for one warp
         (1, 5, 11, 0),   # 67: four warps
         (1, 5, 16, 0),   # 82
         (2, 5, 1, 3),    # 80: the last of 5 rows of blocks, P2
         (1, 6, 1, 3),    # 78
         (1, 6, 8, 1),    # 114: eight warps
         (1, 7, 1, 3),    # 142
         (1, 7, 1, 4),    # 145: sixteen warps
         (2, 6, 1, 4),    # 147
         (2, 7, 1, 0)]    # no frontal kernel: the window in global memory


@pytest.mark.parametrize("P,r,m,l", CASES)
def test_blocks_vs_oracle_at_layout_edges(P, r, m, l):
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


# M up to 64: meshes of more than three elements per SM take one warp per element
@pytest.mark.parametrize("P,r,m,l", [c for c in CASES if 3 * c[2] * (c[3] + 1) + 1 + c[0] * 2 ** c[1] + 2 * c[0] - 1 <= 64])
def test_one_warp_per_element(P, r, m, l):
    """A mesh of more than three elements per SM in one call (one warp per element): blocks and
    reconstruction of some elements against the oracle, and the blocks the same bits as in
    waves of fewer elements (four warps per element)."""
    from paper_1703_10435_gb300.pipeline import Pipeline
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    nx = int(np.ceil(np.sqrt(1.5 * nsm))) + 1   # 2 nx^2 > 3 nsm elements, nx^2 fewer
    w = W.Workload("t", nx, nx, r, P, m, l, "log_uniform", "sinsin", 1.0, 1.0, seed=3)
    kap = W.kappa_for(w) ** 0.25   # contrast 10
    src = mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 1.0)
    p = Pipeline.for_workload(w, 0, mhm.MHM_FP64)
    p.local(torch.as_tensor(kap, device="cuda"), src)
    torch.cuda.synchronize()
    assert int(p.status.abs().sum()) == 0
    full = p.blocks()
    rng = np.random.default_rng(7)
    lam, u0 = rng.standard_normal(p.mesh.n_lambda), rng.standard_normal(2 * nx * nx)
    p.lam, p.u0 = torch.as_tensor(lam, device="cuda"), torch.as_tensor(u0, device="cuda")
    u, _ = p.reconstruct(torch.as_tensor(kap, device="cuda"), src)
    u = u.cpu().numpy()
    mesh = build_mesh(nx, nx, m, l)
    for K in (0, nx * nx, 2 * nx * nx - 1):
        o = solve_local(mesh, K, r, P, kap[K], source_fn("sinsin", 1.0, 1.0))
        tol = max(1e-10, 10 * 1.1e-16 * 12 * o.sub.n * 10)   # 10 u cond, as above
        assert_blocks(*(b[K] for b in full), o, tol, K)
        want = u0[K] + o.eta[:, :-1] @ lam[mesh.local_lambda(K)] + o.eta[:, -1]
        assert np.abs(u[K] - want).max() < tol * np.abs(want).max(), K
    for t in (p.AK, p.EK, p.BK, p.FK):
        t.zero_()
    assert p.local_waves(kap, src, 2 * 8 * 4 ** r * nx * nx) >= 2
    for a, b in zip(full, p.blocks()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("P,r,m", [(1, 1, 1), (1, 2, 1), (2, 1, 4), (1, 3, 1), (2, 2, 4), (1, 3, 4)])
def test_3d_one_warp_and_few_elements_agree(P, r, m):
    """648 tetrahedra in one call (one warp per element) against ranges of 324 (four warps per
    element where the front has room): the same bits."""
    M = mhm.Mesh3D(3, r, P, m, device=0)
    kappa = 10.0 ** torch.as_tensor(np.random.default_rng(5).uniform(-1, 1, (M.n_K, 8 ** r)), device="cuda")
    src = mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0)
    outs = []
    for ranges in (((0, 0),), ((0, 324), (324, 648))):
        f64 = dict(dtype=torch.float64, device="cuda")
        o = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
             torch.zeros(M.n_K, **f64), torch.full((M.n_K,), -7, dtype=torch.int32, device="cuda")]
        for K0, K1 in ranges:
            mhm.mhm3d_local_solve_batch(M, kappa, src, *o, K0=K0, K1=K1)
        outs.append(o)
    assert int(outs[0][4].abs().sum()) == 0 and float(outs[0][0].abs().max()) > 0
    assert all(torch.equal(a, b) for a, b in zip(*outs))


@pytest.mark.parametrize("P,r,m,l", [(1, 0, 1, 0), (1, 3, 1, 1), (1, 4, 2, 0), (2, 4, 3, 1), (1, 5, 2, 2), (1, 6, 1, 3),
                                     (2, 5, 1, 2), (1, 7, 1, 3), (2, 6, 1, 1)])
def test_reconstruction_vs_oracle_at_layout_edges(P, r, m, l):
    """u of both elements from given multipliers (fronts of 3 to 131 slots) against the oracle's
    local solutions combined with the same multipliers."""
    from paper_1703_10435_gb300.pipeline import Pipeline
    w = W.Workload("t", 1, 1, r, P, m, l, "log_uniform", "sinsin", 1.0, 1.0, seed=3)
    kap = W.kappa_for(w) ** 0.25
    src = mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 1.0)
    p = Pipeline.for_workload(w, 0, mhm.MHM_FP64)
    rng = np.random.default_rng(7)
    lam, u0 = rng.standard_normal(p.mesh.n_lambda), rng.standard_normal(2)
    p.lam, p.u0 = torch.as_tensor(lam, device="cuda"), torch.as_tensor(u0, device="cuda")
    u, _ = p.reconstruct(torch.as_tensor(kap, device="cuda"), src)
    u = u.cpu().numpy()
    mesh = build_mesh(1, 1, m, l)
    for K in range(2):
        o = solve_local(mesh, K, r, P, kap[K], source_fn("sinsin", 1.0, 1.0))
        want = u0[K] + o.eta[:, :-1] @ lam[mesh.local_lambda(K)] + o.eta[:, -1]
        tol = max(1e-10, 10 * 1.1e-16 * 12 * o.sub.n * 10)   # 10 u cond, as above
        assert np.abs(u[K] - want).max() < tol * np.abs(want).max(), K


@pytest.mark.parametrize("P,r,m", [(2, 2, 4), (2, 1, 1), (1, 3, 4)])
def test_3d_mixed_on_large_meshes_is_the_fp64_path(P, r, m):
    """MIXED on a mesh of 512 elements or more with room to refine runs the FP64 elimination (the
    same bits, iters 1); one pass or no re-solve runs the refinement, whose blocks agree with it
    to the mixed tolerance."""
    M = mhm.Mesh3D(3, r, P, m, device=0)   # 648 elements
    kappa = 10.0 ** torch.as_tensor(np.random.default_rng(5).uniform(-1, 1, (M.n_K, 8 ** r)), device="cuda")
    src = mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0)

    def run(precision, opts=None):
        f64 = dict(dtype=torch.float64, device="cuda")
        o = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
             torch.zeros(M.n_K, **f64), torch.full((M.n_K,), -7, dtype=torch.int32, device="cuda"),
             torch.full((M.n_K,), -7, dtype=torch.int32, device="cuda")]
        mhm.mhm3d_local_solve_batch(M, kappa, src, *o[:5], precision=precision, opts=opts, iters=o[5])
        return o
    ref, default, explicit = run(mhm.MHM_FP64), run(mhm.MHM_MIXED), run(mhm.MHM_MIXED, mhm.Opts3D(8, 1e-9, 0))
    for got in (default, explicit):
        assert all(torch.equal(a, b) for a, b in zip(ref, got)) and bool((got[5] == 1).all())
    mixed = run(mhm.MHM_MIXED, mhm.Opts3D(8, 1e-9, 1))
    assert int(mixed[4].abs().sum()) == 0 and int(mixed[5].min()) >= 2
    d = ref[0].diagonal(dim1=1, dim2=2).abs().sqrt()
    assert float(((mixed[0] - ref[0]).abs() / (d[:, :, None] * d[:, None]).clamp_min(1e-300)).max()) < 1e-9
    assert float((mixed[1] - ref[1]).abs().max()) < 1e-9 * float(ref[1].abs().max())
