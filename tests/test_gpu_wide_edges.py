"""Mixed precision above rank 32 off the tensor-core path, and the FR-Nys output pass, at the edges of their tiles:
against the float64 oracle at the path's bar (1e-5 on L and S, relative to L), and S + L = M.  Rows on and off 16-byte
boundaries, a last row block of one row, one column tile and several, ranks that fill a group of four and that do not,
more row blocks than CTAs; for FR-Nys odd widths, more ranks than one chunk, and float64 outputs."""
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


def _dev(prob):
    if prob.M.dtype == np.uint16:
        return torch.from_numpy(prob.M.view(np.int16)).view(torch.bfloat16).cuda()
    return torch.from_numpy(prob.M).cuda()


@pytest.mark.parametrize("m,n,r,dtype", [
    (449, 320, 33, "bf16"), (641, 648, 48, "bf16"), (640, 260, 40, "f32"), (961, 700, 63, "f32"), (833, 768, 64, "f32"),
    (300, 333, 37, "f32"), (20000, 256, 34, "f32"), (9901, 132, 33, "f32"),
])
def test_wide_rank_off_tensor_cores_matches_oracle(ctx, m, n, r, dtype):
    prob = synth.planted(m, n, r, p=0.02, amp=50.0, seed=3 * m + n + r, dtype=dtype)
    kw = dict(rho=1.5, mu0=0.05, tol=1e-9, max_iter=300)
    ref = O.fr_adm(prob.values_f64(), r, **kw)
    sol = B.solve_torch(ctx, _dev(prob), r, precision=B.PREC_MIXED, s_dtype=B.F32, want_L=True, **kw)
    assert sol.path == 0
    scale = np.linalg.norm(ref.L)
    assert np.linalg.norm(sol.L.double().cpu().numpy() - ref.L) <= TOL * scale
    assert np.linalg.norm(sol.S.double().cpu().numpy() - ref.S) <= TOL * scale


@pytest.mark.parametrize("m,n,r,l,store,s_dtype", [
    (401, 307, 4, 41, "f32", "F32"), (65, 130, 3, 30, "bf16", "F32"), (256, 256, 5, 64, "bf16", "F64"),
    (700, 516, 33, 264, "f32", "F32"), (449, 387, 40, 301, "f32", "F64"),
])
def test_frnys_output_edges(ctx, m, n, r, l, store, s_dtype):
    prob = synth.planted(m, n, r, p=0.03, amp=1.0, seed=m + n + r, dtype=store)
    perm = torch.from_numpy(synth.row_permutation(m, 17)).cuda()
    sol = B.solve_torch(ctx, _dev(prob), r, nys_l=l, nys_perm=perm, rho=1.5, mu0=0.1, tol=1e-7, max_iter=300,
                        precision=B.PREC_MIXED, s_dtype=getattr(B, s_dtype), want_L=True)
    M = prob.values_f64()
    L, S = sol.L.double().cpu().numpy(), sol.S.double().cpu().numpy()
    U, Bm, V = (x.double().cpu().numpy() for x in (sol.U, sol.B, sol.V))
    exact = U @ Bm @ V.T
    # operands rounded to float32, r products and sums of at most |row of U B| |row of V|: (r + 2) 2^-24, doubled
    bound = (r + 2) * 2.0 ** -23 * np.linalg.norm(U @ Bm, axis=1).max() * np.linalg.norm(V, axis=1).max()
    assert np.abs(L - exact).max() <= bound
    assert np.abs(S + L - M).max() <= 2.0 ** -22 * np.abs(M).max() + 2.0 ** -22 * np.abs(L).max()
