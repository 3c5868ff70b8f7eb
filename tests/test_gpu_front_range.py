"""The FP64 elimination at the ends of the exponent range: kappa times a power of two gives the
blocks and the reconstruction of the unscaled kappa over that power bit for bit (every operation is
exact under a power of two as long as nothing over- or underflows), also where kappa or 1 / kappa is
subnormal, and where one element holds both ends."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_10435_gb300 import mhm

pytestmark = pytest.mark.gpu

# kappa is 2^-3 .. 2^3 times 2^e.  Up: a pivot sums six kappa with weights up to 4, and 2^1024 is
# infinite; down: kappa is exact also where it is subnormal, and the solutions, at most
# |face| / kappa, stay finite
POWERS = [-1022, -1019, -1000, -901, -850, 850, 901, 1000, 1014]


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10435_gb300 import build
    build.build()


def _kappa(shape, seed):
    return np.exp2(np.random.default_rng(seed).integers(-3, 4, shape).astype(float))


@pytest.mark.parametrize("P,r,nx", [(1, 0, 16), (1, 3, 16), (2, 2, 16), (1, 5, 16), (1, 6, 16), (2, 6, 16), (1, 3, 20)])
def test_blocks_and_reconstruction_scale_with_kappa(P, r, nx):
    """nx = 16: up to 16 warps per element; nx = 20 (800 elements): one."""
    from paper_1703_10435_gb300.pipeline import Pipeline
    p = Pipeline(nx, nx, r, P, 1, 1, 0, mhm.MHM_FP64)
    kap = _kappa((2 * nx * nx, 4 ** r), 3)
    src = mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 1.0)
    rng = np.random.default_rng(7)
    p.lam = torch.as_tensor(0.1 * rng.standard_normal(p.mesh.n_lambda), device="cuda")
    p.u0 = torch.zeros(p.mesh.n_K, dtype=torch.float64, device="cuda")

    def solve(k):
        kd = torch.as_tensor(k, device="cuda")
        p.status.fill_(-7)
        p.local(kd, src)
        u, _ = p.reconstruct(kd, src)
        assert int(p.status.abs().sum()) == 0
        return [x.copy() for x in p.blocks()] + [u.cpu().numpy()]
    ref = solve(kap)
    for e in POWERS:
        got = solve(kap * 2.0 ** e)
        # (the mean of u sums mass times u: above 2^1000 those are subnormal)
        for k, (a, b) in enumerate(zip(ref, got if e <= 1000 else got[:4])):
            want = a if k in (2, 3) else np.ldexp(a, -e)   # B_K and F_K do not depend on kappa
            # (a subnormal value is rounded to a multiple of 2^-1074)
            assert np.all(np.abs(b - want) <= (0.0 if e < 850 else 2.0 ** -1074)), (e, k)


def test_both_ends_in_one_element():
    """One fine triangle (inside) at 2^-1000 in an element at 2^100: solved, finite, and as with
    2^-400 there, which couples as little next to 2^100."""
    from paper_1703_10435_gb300.pipeline import Pipeline
    p = Pipeline(2, 2, 3, 1, 1, 1, 0, mhm.MHM_FP64)
    kap = np.full((8, 64), 2.0 ** 100)
    src = mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 1.0)
    out = []
    for soft in (2.0 ** -1000, 2.0 ** -400):
        kap[:, 20] = soft
        p.local(torch.as_tensor(kap, device="cuda"), src)
        torch.cuda.synchronize()
        assert int(p.status.abs().sum()) == 0
        out.append([x.copy() for x in p.blocks()])
    for a, b in zip(*out):
        assert np.all(np.isfinite(a)) and np.abs(a - b).max() <= 1e-12 * np.abs(a).max()


@pytest.mark.parametrize("nc,r,P,m", [(1, 1, 2, 4), (3, 1, 2, 4), (1, 2, 2, 16)])
@pytest.mark.parametrize("precision", [mhm.MHM_FP64, mhm.MHM_MIXED])
def test_3d_blocks_scale_with_kappa(nc, r, P, m, precision):
    """MIXED cannot refine in FP32 here and ends with the FP64 blocks."""
    M = mhm.Mesh3D(nc, r, P, m)
    kap = _kappa((M.n_K, 8 ** r), 5)
    f64 = dict(dtype=torch.float64, device="cuda")
    o = [torch.zeros(M.n_K, M.n_I, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64), torch.zeros(M.n_K, M.n_I, **f64),
         torch.zeros(M.n_K, **f64), torch.zeros(M.n_K, dtype=torch.int32, device="cuda")]

    def solve(k, prec):
        o[4].fill_(-7)
        mhm.mhm3d_local_solve_batch(M, torch.as_tensor(k, device="cuda"), mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, 2.0),
                                    *o, precision=prec)
        assert int(o[4].abs().sum()) == 0
        return [x.cpu().numpy() for x in o[:4]]
    ref = solve(kap, mhm.MHM_FP64)
    for e in (-1018, -1000, 901, 1000, 1016):
        for k, (a, b) in enumerate(zip(ref, solve(kap * 2.0 ** e, precision))):
            want = a if k in (2, 3) else np.ldexp(a, -e)
            if precision == mhm.MHM_FP64 or m > 4 or M.n_K >= 512:
                assert np.all(np.abs(b - want) <= (0.0 if e < 850 else 2.0 ** -1074)), (e, k)
            else:   # a refined element: the mixed tolerance
                assert np.abs(b - want).max() <= 1e-9 * np.abs(want).max(), (e, k)
