"""Float64 results of matrices whose rows or columns differ in size by up to 1e10, neighbours in one tile of the kernels:
each row (column) has to be as accurate as its own size allows, as float64 multiply-add loops leave it, whatever
stands beside it.  Against the float64 oracle, row by row: a row of U and of L = U B V^T is a sum of products of that row
alone with factors shared by all rows, whose errors (1e-13 and below at these condition numbers) are relative to the row."""
import numpy as np
import pytest

from oracle import fradm as O
from paper_1503_03004_gb300 import binding as B

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROW_TOL = 1e-11


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = B.Context(0)
    yield c
    c.close()


def _scales(k, seed):
    """Half of them 1, the others 1e-10 .. 1 in random order, the first and last of each 64 the largest and the smallest."""
    rng = np.random.default_rng(seed)
    s = 10.0 ** -np.where(rng.random(k) < 0.5, 0.0, rng.uniform(0, 10, k))
    s[::64], s[63::64] = 1.0, 1e-10
    return s


def _low_rank(m, n, r, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((m, r)) @ rng.standard_normal((r, n))


def _row_error(A, R):
    return (np.linalg.norm(A - R, axis=1) / np.linalg.norm(R, axis=1)).max()


@pytest.mark.parametrize("r", [5, 12, 30, 50])
def test_truncated_svd_rows_of_different_size(ctx, r):
    # (12 steps: from the nearly dependent first 30 columns the factors take about ten to settle)
    m, n = 333, 260
    M = _scales(m, r)[:, None] * _low_rank(m, n, r, r)
    Ur, Br, Vr = O.fixed_rank_opt_full(M, np.eye(m, r), np.eye(r), np.eye(n, r), 12)[-1]
    sol = B.opt_full_torch(ctx, torch.from_numpy(M).cuda(), r, tol=0.0, max_iter=12, precision=B.PREC_FP64)
    L = (sol.U @ sol.B @ sol.V.T).cpu().numpy()
    assert _row_error(L, Ur @ Br @ Vr.T) <= ROW_TOL


def _planted(m, n, r, seed):
    """Low rank with independent first r columns, plus outliers of five times the entries' size on 5 % of them."""
    rng = np.random.default_rng(seed)
    R = rng.standard_normal((r, n))
    R[:, :r] = np.sqrt(r) * np.linalg.qr(R[:, :r])[0]
    S = np.where(rng.random((m, n)) < 0.05, rng.uniform(-5, 5, (m, n)) * np.sqrt(r), 0.0)
    return rng.standard_normal((m, r)) @ R + S


# The path's own bar (1e-9 in norm), here for each row or column in its own size.
@pytest.mark.parametrize("m,n,r", [(333, 260, 5), (300, 321, 12), (400, 260, 24), (390, 330, 50), (2100, 96, 8)])
def test_robust_rows_of_different_size(ctx, m, n, r):
    M = _scales(m, r)[:, None] * _planted(m, n, r, 10 + r)
    ref = O.fr_adm(M, r, rho=1.5, mu0=0.1, fixed_iters=12)
    sol = B.solve_torch(ctx, torch.from_numpy(M).cuda(), r, fixed_iters=12, rho=1.5, mu0=0.1)
    assert _row_error((sol.U @ sol.B @ sol.V.T).cpu().numpy(), ref.L) <= 1e-9


@pytest.mark.parametrize("m,n,r", [(260, 333, 5), (321, 300, 12), (260, 400, 24), (330, 390, 50), (96, 2100, 8)])
def test_robust_columns_of_different_size(ctx, m, n, r):
    s = _scales(n, r)
    s[:r] = 1.0  # (the iteration starts from the first r columns)
    M = s[None, :] * _planted(m, n, r, 10 + r)
    ref = O.fr_adm(M, r, rho=1.5, mu0=0.1, fixed_iters=12)
    sol = B.solve_torch(ctx, torch.from_numpy(M).cuda(), r, fixed_iters=12, rho=1.5, mu0=0.1)
    assert _row_error((sol.U @ sol.B @ sol.V.T).cpu().numpy().T, ref.L.T) <= 1e-9
