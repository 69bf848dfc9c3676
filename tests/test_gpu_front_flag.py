"""Whether a flow has a front is found anew by each call: a call's result does not depend on the flow
that an earlier call on the same context saw."""
import numpy as np
import pytest

from paper_2410_05489_gb300 import problems as P
from test_gpu_parity import A, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [5, 9])
def test_a_step_after_a_step_adjoint_of_a_front(A, order):  # noqa: F811
    import torch

    pb, Wf = P.riemann_2d(160, order, 17 + order)
    front, fresh = A.Solver(pb, Wf), A.Solver(pb)
    smooth = P.smooth_random(pb.replace(bc=("periodic",) * 4), order)
    try:
        front.step()  # strengths of the fronts, and a dt that the state carries
        _, dt, _ = front.status()
        bars = [torch.ones_like(t) for t in (front.W, front.sx, front.sy)]
        front.step_adjoint(front.W, front.sx, front.sy, 0.5 * dt, *bars)
        for s in (front, fresh):
            s.W.copy_(to_dev(smooth))
            s.prime()
            s.step(1e-4 * dt)
        lim = pb.sigma_thres / 16.0
        assert float(fresh.sx.max()) < lim or float(fresh.sy.max()) < lim  # no front in one direction
        for a, b in zip((front.W, front.sx, front.sy), (fresh.W, fresh.sx, fresh.sy)):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    finally:
        front.close()
        fresh.close()
