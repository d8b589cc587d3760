"""Mixed precision above rank 32 off the tensor-core path, where a thin sum runs over thousands of columns (Q, one column
split) or rows (W): each tile's sum is formed by itself and then added.  A planted L is recovered exactly (the solve
converges to 1e-9), so the error of L is the path's own float32 rounding.  Bar: sums in 64-column tiles and over 64 of them
round like sqrt(64) + sqrt(64) units of 2^-24, 1.0e-6, in Q and about as much in W, and the product U C^T like
sqrt(40), 0.4e-6: 1.5e-6 together, doubled; one chain over 4096 columns and 8000 rows would be at sqrt(4096) and sqrt(8000)
units, 6.5e-6."""
import pytest

from paper_1503_03004_gb300 import binding as B

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n,r", [(40000, 4096, 40), (8192, 16384, 40)])
def test_error_of_long_float32_sums(m, n, r):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    g = torch.Generator("cuda").manual_seed(m + n + r)
    U0, V0 = (torch.randn((k, r), generator=g, device="cuda", dtype=torch.float64) for k in (m, n))
    M = torch.rand((m, n), generator=g, device="cuda").mul_(100).sub_(50)
    M.mul_(torch.rand((m, n), generator=g, device="cuda") < 0.05)
    M = M.addmm_(U0.float(), V0.float().T)
    with B.Context(0) as ctx:
        sol = B.solve_torch(ctx, M, r, precision=B.PREC_MIXED, s_dtype=B.F32, want_L=True, mu0=0.05, rho=1.5, tol=1e-9,
                            max_iter=300)
    L0 = U0 @ V0.T
    assert sol.path == 0
    assert float((sol.L - L0).norm() / L0.norm()) <= 3e-6
