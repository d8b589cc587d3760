"""Float64 requests of different ranks in one padded-rank class, solved at the same time by the serving slots' threads,
long enough to run the fixed-point kernels above rank 16 too (their shared memory follows the rank; the first six
iterations there are float64 loops).  Each has to end as it does alone."""
import numpy as np
import pytest

from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("lo,hi", [(17, 32), (33, 64)])
def test_concurrent_ranks_above_16_equal_solo_solves(lo, hi):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with B.Context(0) as ctx:
        todo, keep = [], []
        for i in range(24):
            r = lo + (5 * i) % (hi - lo + 1)
            p = synth.planted(300 + 13 * i, (260, 321, 200)[i % 3], r, p=0.05, amp=1.0, seed=700 + i, dtype="f64")
            M = torch.from_numpy(np.ascontiguousarray(p.M)).cuda()
            todo.append((M, r, B.solve_torch(ctx, M, r, fixed_iters=12)))
        for M, r, _ in todo:
            m, n = M.shape
            S = torch.empty((m, n), dtype=torch.float64, device="cuda")
            prob = B.make_problem(m=m, n=n, r=r, M_ptr=M.data_ptr(), m_dtype=B.F64, fixed_iters=12)
            res = B.make_result(S_ptr=S.data_ptr(), s_dtype=B.F64, lds=n)
            keep.append((S, prob, res, ctx.submit(prob, res)))
        assert [ctx.poll(k[3], -1) for k in keep] == [B.OK] * len(keep)
        for (_, _, alone), (S, _, _, _) in zip(todo, keep):
            assert torch.equal(S, alone.S)
