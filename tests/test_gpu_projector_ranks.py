"""The r x r projector at ranks that are not multiples of 4: its float32 products are padded to the next multiple with
zeros, so a call takes no longer than at that multiple (a tail of the sums and a second store path made r = 38
slower than r = 40).  Times are the library's own, averaged over the calls of a solve, the two ranks in turn, medians of
five; 3 % are left for calls that settle earlier or later."""
import numpy as np
import pytest

from paper_1503_03004_gb300 import binding as B
from paper_1503_03004_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _call_us(r):
    """Mean time of a projector call of one solve of 60 iterations, most of them settled."""
    prob = synth.planted(1536, 1024, r, p=0.05, amp=50.0, seed=5, dtype="bf16")
    M = torch.from_numpy(prob.M.view(np.int16)).view(torch.bfloat16).cuda()
    kw = dict(precision=B.PREC_MIXED, s_dtype=B.F32, fixed_iters=60, rho=1.4, mu0=0.05)
    with B.Context(0, profile=1) as ctx:
        B.solve_torch(ctx, M, r, **kw)
        ctx.stats(reset=True)
        B.solve_torch(ctx, M, r, **kw)
        s = ctx.stats()[B.STAT_RXR]
        return 1e3 * s["total_ms"] / s["timed"]


@pytest.mark.parametrize("r", [37, 38, 46])
def test_projector_call_no_slower_than_at_the_next_multiple_of_4(r):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    r4 = (r + 3) // 4 * 4
    odd, even = (float(np.median(x)) for x in zip(*[(_call_us(r), _call_us(r4)) for _ in range(5)]))
    print(f"r = {r}: {odd:.1f} us a call, r = {r4}: {even:.1f} us")
    assert odd <= 1.03 * even
