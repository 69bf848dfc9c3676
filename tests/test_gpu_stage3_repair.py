"""The positivity repair of the third stage, whose result overwrites W^n: steps in which it acts against
the oracle, one step at a time, and the batch against the same problem alone."""
import numpy as np
import pytest

from parity_report import check
from paper_2410_05489_gb300 import problems as P
from test_gpu_parity import A, TOL_STEPS, comp_err  # noqa: F401

pytestmark = pytest.mark.gpu


def streams(ndim, n, order):
    """Two streams that leave each other at Mach ~40 on a periodic box (2D: along an oblique line)."""
    pb = P.Problem(ndim=ndim, nx=n, ny=n if ndim == 2 else 1, order=order, bc=("periodic",) * 4)
    x = (np.arange(n) + 0.5) / n
    if ndim == 1:
        left, v = (x < 0.5)[None, :], ()
    else:
        X, Y = np.meshgrid(x, x)
        left = (X + 0.3 * Y) % 1.0 < 0.5
        v = (np.where(left, -1.8, 1.8),)
    prim = (np.ones(left.shape), np.where(left, -6.0, 6.0), *v, np.full(left.shape, 0.02))
    return pb, np.ascontiguousarray(P.conservative(prim, pb.gamma, ndim))


@pytest.mark.parametrize("case", [(1, 100, 5, 42), (2, 40, 5, 18), (2, 40, 7, 18), (2, 40, 9, 18)])
def test_third_stage_repair_parity(A, oracle, case):  # noqa: F811
    ndim, n, order, steps = case
    pb, W0 = streams(ndim, n, order)
    s = A.Solver(pb, W0)
    acted = 0
    try:
        for _ in range(steps):
            W, sx, sy = (t.cpu().numpy() for t in (s.W, s.sx, s.sy))
            s.step()
            if A.ase_df_get_repair_stats(s.ctx)[0][0] == 0:  # cells marked in the last stage
                continue
            acted += 1
            Wc = oracle.step(pb, W, sx, sy, s.status()[1])[0]
            check("W after a step", comp_err(s.W.cpu().numpy(), Wc), TOL_STEPS)
    finally:
        s.close()
    assert acted > 0


def test_batch_repairs_the_third_stage_alike(A):  # noqa: F811
    from paper_2410_05489_gb300 import batch

    probs = [streams(2, 40, 5), streams(1, 100, 5)]
    bt = batch.Batch([p for p, _ in probs], [w for _, w in probs])
    try:
        bt.run(42)
        for i, (pb, W) in enumerate(probs):
            s = A.Solver(pb, W)
            s.run(42)
            assert np.array_equal(bt.state(i), s.W.cpu().numpy())
            s.close()
    finally:
        bt.close()
