"""1D problems at the edges of their tiles (31 faces) and of the launch that combines and repairs in one
CTA (416 cells): the steps of the batch, whose 255-face tiles and separate launches do the same arithmetic."""
import numpy as np
import pytest

from parity_report import check
from paper_2410_05489_gb300 import problems as P
from test_gpu_parity import A, TOL_STEPS, comp_err  # noqa: F401

pytestmark = pytest.mark.gpu

SIZES = [9, 29, 30, 31, 41, 42, 61, 62, 63, 93, 255, 415, 416, 417, 1000]


@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_steps_equal_the_batch(A, oracle, order):  # noqa: F811
    from paper_2410_05489_gb300 import batch

    probs = [P.riemann_1d(n, order, 13 * order + n) for n in SIZES]
    probs += [P.sin_wave_1d(n, order) for n in SIZES]
    bt = batch.Batch([p for p, _ in probs], [w for _, w in probs])
    try:
        bt.run(3)
        for i, (pb, W) in enumerate(probs):
            s = A.Solver(pb, W)
            s.run(3)
            assert np.array_equal(bt.state(i), s.W.cpu().numpy()), pb.nx
            assert np.array_equal(bt.sigma(i)[0], s.sx.cpu().numpy()), pb.nx
            if pb.nx in (31, 417):
                check("W vs oracle", comp_err(s.W.cpu().numpy(), oracle.run(pb, W, nsteps=3)[0]), TOL_STEPS, i)
            s.close()
    finally:
        bt.close()
