"""Float64 path at the edges of its tiles and rank groups: 32-row sweep blocks, 64-column tiles, 4 x 2
output units with the sums split over up to 32 groups, every padded rank, odd widths, float32 and
bfloat16 storage, wide and tall shapes (several row chunks and column splits), and ranks above 32, whose
first iterations run float64 loops before the fixed-point kernels take over.  Against the float64
oracle at the path's bar (1e-9 on L, B and S in L's scale, fixed before the first run)."""
import numpy as np
import pytest

from oracle import fradm as O
from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-9


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    c = B.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("m,n,r,dtype", [
    (33, 129, 1, "f64"), (64, 64, 2, "f32"), (65, 63, 5, "bf16"), (31, 200, 8, "f64"), (95, 97, 9, "f64"),
    (128, 321, 12, "bf16"), (300, 70, 13, "f32"), (127, 190, 16, "f64"), (257, 130, 17, "f64"), (96, 1000, 28, "f32"),
    (1400, 100, 32, "bf16"), (200, 190, 33, "f64"), (129, 300, 47, "f32"), (333, 140, 64, "bf16"),
    (4000, 66, 3, "f64"), (70, 5000, 4, "f64"),
])
def test_float64_edges_match_oracle(ctx, m, n, r, dtype):
    prob = synth.planted(m, n, r, p=0.05, amp=5.0, seed=3 * m + n + r, dtype=dtype)
    ref = O.fr_adm(prob.values_f64(), r, rho=1.5, mu0=0.1, fixed_iters=10)
    M = torch.from_numpy(prob.M.view(np.int16)).view(torch.bfloat16) if dtype == "bf16" else torch.from_numpy(prob.M)
    sol = B.solve_torch(ctx, M.cuda(), r, fixed_iters=10, rho=1.5, mu0=0.1)
    scale = np.linalg.norm(ref.L)
    L = (sol.U @ sol.B @ sol.V.T).cpu().numpy()
    assert np.linalg.norm(L - ref.L) <= TOL * scale
    assert np.linalg.norm(sol.S.cpu().numpy() - ref.S) <= TOL * scale
    np.testing.assert_allclose(sol.B.cpu().numpy(), ref.B, atol=TOL * np.abs(ref.B).max())
