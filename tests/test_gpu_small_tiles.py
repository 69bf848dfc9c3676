"""The sweep's tiles of at most 16 lines (several threads a face: grids below 197^2 cells), and
the rules that keep noise strengths in FP64.

Tiles: against the oracle at the bounds of test_gpu_parity.py (whose small random grids take them
too), on shapes that give tiles of 8 and of 16 lines, ragged last tiles in both directions, thin grids
and (141 x 133) the fixed-point reconstructions; and against the batch's 64-line tiles, which do the
same FP64 arithmetic without a front: the same bits."""
import numpy as np
import pytest

from paper_2410_05489_gb300 import problems as P
from test_gpu_parity import A, check_residual  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(64, 64), (61, 67), (9, 130), (150, 11), (97, 90), (141, 133)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_residual_parity(A, oracle, order, shape):  # noqa: F811
    pb, W = P.riemann_2d(shape[0], order, 11 * order + shape[1], ny=shape[1])
    sx, sy = oracle.prime_sigma(pb, W)
    check_residual(A, oracle, pb, W, sx, sy)


@pytest.mark.parametrize("shape", [(9, 130), (10, 33), (40, 9), (12, 12)])
@pytest.mark.parametrize("order", [5, 7, 9])
def test_walls_on_thin_grids(A, oracle, order, shape):  # noqa: F811
    """A tile wider than the grid stages cells beyond the mirrored ones."""
    pb, W = P.riemann_2d(shape[0], order, 5 * order + shape[1], ny=shape[1])
    pb = pb.replace(bc=("reflect",) * 4)
    sx, sy = oracle.prime_sigma(pb, W)
    check_residual(A, oracle, pb, W, sx, sy)


@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_strengths_equal_the_batch_tiles(A, order):  # noqa: F811
    from paper_2410_05489_gb300 import batch

    probs = [P.isentropic_vortex(n, order, ny=m) for n, m in ((64, 64), (61, 67), (97, 90))]
    bt = batch.Batch([p for p, _ in probs], [w for _, w in probs])
    try:
        for i, (pb, W) in enumerate(probs):
            s = A.Solver(pb, W)
            for got, ref in zip(bt.sigma(i), (s.sx, s.sy)):
                assert np.array_equal(got, ref.cpu().numpy())
            s.close()
    finally:
        bt.close()


@pytest.mark.parametrize("flow", ["fast", "one direction"])
@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_noise_strengths_keep_their_bits(A, order, flow):  # noqa: F811
    """Strengths that are the rounding of the states: a fast stream (pressure 1e-6 of its energy), and a
    slow one with a front across one direction only.  A strength of 1 elsewhere in the grid (below
    sigma_thres: no branch changes) must not turn fixed point on in these tiles."""
    import torch

    n = 256
    pb = P.Problem(ndim=2, nx=n, ny=n, order=order, bc=("periodic",) * 4)
    rng = np.random.default_rng(order)
    one = np.ones((n, n))
    u = 800.0 if flow == "fast" else 0.5
    W = P.conservative((5.0 * one, u * one, 0.0 * one, 0.4 * (1.0 + 0.01 * rng.random((n, n)))), pb.gamma, 2)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    sx, sy = np.zeros(pb.sx_shape), np.zeros(pb.sy_shape)
    s = A.Solver(pb)
    try:
        ref = [t.cpu().numpy() for t in s.residual(dev(W), dev(sx), dev(sy))]
        sx[128, 128] = 1.0
        if flow == "fast":
            sy[40, 200] = 1.0
        got = [t.cpu().numpy() for t in s.residual(dev(W), dev(sx), dev(sy))]
    finally:
        s.close()
    for a, b in zip(got, ref):
        assert np.array_equal(a, b)
