"""Mixed-precision SIMT passes (r <= 32) at the edges of their tiles, against the float64 oracle at the path's bar
(1e-5 on L and S, relative to L): narrow matrices whose sweep keeps only the needed columns in up to
four stages, widths around one and two 64-column tiles, every padded rank, rows off 16-byte
boundaries, a last row block of one row, and more row blocks than CTAs."""
import numpy as np
import pytest

from oracle import fradm as O
from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-5


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("m,n,r,dtype", [
    (700, 16, 2, "f32"), (65, 24, 1, "bf16"), (1500, 37, 3, "bf16"), (90001, 40, 3, "f32"), (513, 48, 5, "f32"),
    (800, 63, 8, "bf16"), (640, 64, 9, "f32"), (449, 65, 7, "bf16"), (321, 96, 12, "bf16"), (577, 127, 16, "f32"),
    (400, 129, 17, "bf16"), (1025, 200, 25, "f32"), (512, 191, 29, "bf16"), (700, 320, 32, "f32"), (2100, 333, 31, "bf16"),
])
def test_simt_edges_match_oracle(ctx, m, n, r, dtype):
    prob = synth.planted(m, n, r, p=0.04, amp=50.0, seed=5 * m + n + r, dtype=dtype)
    kw = dict(rho=1.5, mu0=0.05, tol=1e-9, max_iter=300)
    ref = O.fr_adm(prob.values_f64(), r, **kw)
    M = torch.from_numpy(prob.M.view(np.int16)).view(torch.bfloat16) if dtype == "bf16" else torch.from_numpy(prob.M)
    sol = B.solve_torch(ctx, M.cuda(), r, precision=B.PREC_MIXED, s_dtype=B.F32, want_L=True, **kw)
    assert sol.path == 0 and sol.rel_residual <= 1e-9
    scale = np.linalg.norm(ref.L)
    assert np.linalg.norm(sol.L.double().cpu().numpy() - ref.L) <= TOL * scale
    assert np.linalg.norm(sol.S.double().cpu().numpy() - ref.S) <= TOL * scale
