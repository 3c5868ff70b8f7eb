"""Systems that mhm_solve_global has to refuse: singular ones, ones whose A is not negative definite
in a large front of the dissection, and ones with a pivot that cannot be divided by.  After a
refusal the same mesh solves the proper system again with the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1703_10435_gb300 import mhm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10435_gb300 import build
    build.build()


def _system(nx, m, l, field="log_uniform"):
    from paper_1703_10435_gb300.pipeline import Pipeline
    w = W.Workload("t", nx, nx, 3, 1, m, l, field, "const", 1.0, seed=17)
    p = Pipeline.for_workload(w, 0, mhm.MHM_FP64)
    p.step(torch.as_tensor(W.kappa_for(w), device="cuda").contiguous(), mhm.Source(mhm.MHM_SRC_CONST, 1.0, 1.0))
    rp = p.mesh.query(mhm.Q_CSR_ROWPTR, np.int32, p.mesh.n_lambda + 1)
    co = p.mesh.query(mhm.Q_CSR_COLS, np.int32, p.mesh.nnz)
    diag = np.array([rp[i] + int(np.searchsorted(co[rp[i]:rp[i + 1]], i)) for i in range(p.mesh.n_lambda)])
    assert np.array_equal(co[diag], np.arange(p.mesh.n_lambda))
    return p, p.A_vals.clone(), torch.as_tensor(diag, device="cuda")


def _middle_multipliers(p, nx):
    """Multipliers on the line x = 1/2, the separator at the root of the dissection."""
    M = p.mesh
    kl = M.query(mhm.Q_K_LAMBDA, np.int32, M.n_K * M.n_I).reshape(M.n_K, 3, -1)
    xy = W.coarse_vertices(nx, nx)   # (n_K, 3, 2), face a opposite vertex a
    on = [kl[K, a] for K in range(M.n_K) for a in range(3)
          if np.all(np.abs(xy[K, [(a + 1) % 3, (a + 2) % 3], 0] - 0.5) < 1e-12)]
    assert on
    return np.unique(np.concatenate(on))


def _refused(p):
    with pytest.raises(mhm.MHMError) as e:
        p.solve_global()
    assert e.value.code == mhm.MHM_ERR_INVALID_ARG


def test_indefinite_large_front_refused():
    """40 x 40 squares, six multipliers per face: the root separator's front has 240 rows."""
    p, A, diag = _system(40, 2, 2)
    lam, u0 = (x.clone() for x in p.solve_global())
    p.A_vals.neg_()
    _refused(p)
    for i in _middle_multipliers(p, 40)[[0, 100, -1]]:
        p.A_vals.copy_(A)
        p.A_vals[diag[int(i)]] = 1e6 * float(A.abs().max())
        _refused(p)
    p.A_vals.copy_(A)
    lam2, u02 = p.solve_global()
    assert torch.equal(lam, lam2) and torch.equal(u0, u02)


def test_wrong_sign_in_small_fronts_solved():
    """4 x 4 squares: no front is large.  -A is solved with the same multipliers on the
    homogeneous constraint's complement: [-A B^T; B 0] x = [-E; F] has lambda as before, -u0."""
    p, A, diag = _system(4, 1, 1)
    E = p.E.clone()
    lam, u0 = (x.clone() for x in p.solve_global())
    p.A_vals.neg_()
    p.E.copy_(-E)
    lam2, u02 = p.solve_global()
    # both are backward stable solves of the same system up to signs: 1e-10 as in the other tests
    assert float((lam - lam2).abs().max()) <= 1e-10 * float(lam.abs().max())
    assert float((u0 + u02).abs().max()) <= 1e-10 * float(u0.abs().max())


@pytest.mark.parametrize("nx", [1, 4])
def test_pivots_that_cannot_be_divided_by_refused(nx):
    """Diagonal entries of 2^1021 and more (whose reciprocals reach the subnormals), infinite, NaN,
    and a zero A."""
    p, A, diag = _system(nx, 1, 0, "one")
    lam, u0 = (x.clone() for x in p.solve_global())
    d = A[diag].abs()
    p.A_vals.copy_(A * 2.0 ** 500 * 2.0 ** (521 - int(np.floor(np.log2(float(d.min()))))))
    _refused(p)   # (the first unknown's pivot is its diagonal entry)
    for v in (float("inf"), -float("inf"), float("nan")):
        p.A_vals.copy_(A)
        p.A_vals[diag[0]] = v
        _refused(p)
    p.A_vals.zero_()
    _refused(p)
    p.A_vals.copy_(A)
    lam2, u02 = p.solve_global()
    assert torch.equal(lam, lam2) and torch.equal(u0, u02)
