"""What sfr_stats says of a float64 solve above rank 16, whose first iterations are enqueued one by one: every iteration
that ran is timed once, with the bytes of its own operands (the W pass reads M in iteration 1 and Delta, float64, in the
others), and an iteration that found the stop flag set is not."""
import pytest

from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("r,iters", [(20, 1), (20, 3), (20, 7), (20, 12), (40, 6), (8, 5)])
def test_every_iteration_is_timed_once(r, iters):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m, n = 300, 260
    M = torch.from_numpy(synth.planted(m, n, r, p=0.05, amp=5.0, seed=r + iters, dtype="f32").M).cuda()
    with B.Context(0, profile=1) as ctx:
        sol = B.solve_torch(ctx, M, r, fixed_iters=iters, rho=1.5, mu0=0.1)
        st = ctx.stats()
    assert sol.iters == iters
    assert [st[k]["timed"] for k in (B.STAT_SWEEP, B.STAT_WPASS, B.STAT_RXR)] == [iters, iters, 2 * iters]
    assert st[B.STAT_SWEEP]["bytes"] == m * n * (4 + 3 * 8.0) * iters
    assert st[B.STAT_WPASS]["bytes"] == m * n * (4 + 8.0 * (iters - 1))
    assert all(st[k]["total_ms"] > 0 for k in (B.STAT_SWEEP, B.STAT_WPASS, B.STAT_RXR))
    with B.Context(0, profile=2) as ctx:  # one sweep in four
        B.solve_torch(ctx, M, r, fixed_iters=iters, rho=1.5, mu0=0.1)
        assert 1 <= ctx.stats()[B.STAT_SWEEP]["timed"] <= 1 + iters // 4


@pytest.mark.parametrize("iters", [1, 2, 3, 4, 6])
def test_short_solves_launch_no_idle_iterations(iters):
    # iterations go out in pairs after the first: at most one past the cap
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    M = torch.from_numpy(synth.planted(300, 260, 20, p=0.05, amp=5.0, seed=iters, dtype="f64").M).cuda()
    with B.Context(0, profile=1) as ctx:
        long = B.solve_torch(ctx, M, 20, fixed_iters=12, rho=1.5, mu0=0.1)
        ctx.stats(reset=True)
        short = B.solve_torch(ctx, M, 20, fixed_iters=iters, rho=1.5, mu0=0.1)
        assert ctx.stats()[B.STAT_SWEEP]["launches"] <= iters + 1
        again = B.solve_torch(ctx, M, 20, fixed_iters=12, rho=1.5, mu0=0.1)  # the graphs kept from the first solve
    assert short.iters == iters and torch.equal(again.S, long.S) and torch.equal(again.U, long.U)
    with B.Context(0) as ctx:  # the short solve first: it captures the graphs that the long one runs
        assert torch.equal(B.solve_torch(ctx, M, 20, fixed_iters=iters, rho=1.5, mu0=0.1).U, short.U)
        assert torch.equal(B.solve_torch(ctx, M, 20, fixed_iters=12, rho=1.5, mu0=0.1).U, long.U)
