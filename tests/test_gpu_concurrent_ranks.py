"""Requests of different ranks and widths in one padded-rank class, solved at the same time by the serving slots'
threads: they launch the same kernels with different amounts of shared memory, and each has to end as it does alone."""
import numpy as np
import pytest

from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("store,precision", [("f64", B.PREC_FP64), ("f32", B.PREC_MIXED)])
def test_concurrent_ranks_equal_solo_solves(store, precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    ctx = B.Context(0)
    t = torch.float64 if store == "f64" else torch.float32
    code = B.F64 if store == "f64" else B.F32
    M, alone = [], []
    for i in range(40):
        r = 1 + i % 8 if i % 2 else 17 + i % 16
        p = synth.planted(130 + 7 * i, (48, 96, 260)[i % 3], r, p=0.05, amp=1.0, seed=900 + i, dtype=store)
        M.append((torch.from_numpy(np.ascontiguousarray(p.M)).cuda(), r))
        alone.append(B.solve_torch(ctx, M[-1][0], r, fixed_iters=6, precision=precision, s_dtype=code))
    keep, tickets = [], []
    for Md, r in M:
        m, n = Md.shape
        S = torch.empty((m, n), dtype=t, device="cuda")
        prob = B.make_problem(m=m, n=n, r=r, M_ptr=Md.data_ptr(), m_dtype=code, fixed_iters=6, precision=precision)
        res = B.make_result(S_ptr=S.data_ptr(), s_dtype=code, lds=n)
        keep.append((S, prob, res))
        tickets.append(ctx.submit(prob, res))
    assert [ctx.poll(x, -1) for x in tickets] == [B.OK] * len(tickets)
    for a, (S, _, _) in zip(alone, keep):
        assert torch.equal(S, a.S)
    ctx.close()
