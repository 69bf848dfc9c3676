"""The fixed-point reconstructions of the 2D sweep (grids of 128^2 cells or more whose strengths
hold a front) against the oracle, at the bounds of test_gpu_parity.py: the error of a value is
about 2^-56 of its tile's largest, below an FP64 chain's, so the same bounds hold.

Shapes: ragged tails in both directions, thin grids (a last tile column of 5 faces, blocks of a
few lines), the smallest grid that takes the path.  Data: random quadrants (jumps beyond the
range one exponent serves: tiles in FP64), white noise (every branch), a smooth field with
random strengths (all branches in tiles in range), a tube along x (zero momentum along y),
and the noise on the walls' mirrored ghosts."""
import numpy as np
import pytest

from paper_2410_05489_gb300 import problems as P
from test_gpu_parity import A, check_residual  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(141, 133), (700, 24), (21, 800), (128, 128)]


def data(kind, nx, ny, order, seed):
    if kind == "riemann":
        return P.riemann_2d(nx, order, seed, ny=ny)
    if kind == "tube":
        pb = P.Problem(ndim=2, nx=nx, ny=ny, order=order)
        x = (np.arange(nx) + 0.5) * pb.dx
        left = np.broadcast_to(x < 0.5, (ny, nx))
        z = np.zeros((ny, nx))
        return pb, np.ascontiguousarray(P.conservative((np.where(left, 1.0, 0.125), z, z, np.where(left, 1.0, 0.1)),
                                                       pb.gamma, 2))
    bc = ("reflect", "reflect", "outflow", "reflect") if kind == "walls" else ("periodic",) * 4
    pb = P.Problem(ndim=2, nx=nx, ny=ny, order=order, bc=bc)
    return pb, P.smooth_random(pb, seed) if kind == "smooth" else P.white_noise(pb, seed)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["riemann", "noise", "smooth", "tube", "walls"])
@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_front_residual_parity(A, oracle, order, kind, shape):  # noqa: F811
    pb, W = data(kind, shape[0], shape[1], order, 7 * order + shape[0])
    if kind in ("riemann", "tube"):
        sx, sy = oracle.prime_sigma(pb, W)
    else:
        sx, sy = P.random_sigma(pb, order, 1.0)  # stencil sums straddle sigma_thres = 2
    assert max(sx.max(), sy.max()) > pb.sigma_thres / 16.0
    check_residual(A, oracle, pb, W, sx, sy)


def test_non_finite_value_takes_the_first_order_point(A, oracle):  # noqa: F811
    """A NaN cell in a front flow puts its tiles on the FP64 path; cells away from it keep their values."""
    import torch

    pb, W = P.riemann_2d(160, 7, 5, ny=128)
    sx, sy = oracle.prime_sigma(pb, W)
    s = A.Solver(pb)
    try:
        dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
        clean = [t.cpu().numpy() for t in s.residual(dev(W), dev(sx), dev(sy))]
        Wn = W.copy()
        Wn[3, 60, 80] = np.nan
        out = [t.cpu().numpy() for t in s.residual(dev(Wn), dev(sx), dev(sy))]
    finally:
        s.close()
    far = np.ones((128, 160), bool)
    far[60 - 9:60 + 10, 80 - 9:80 + 10] = False
    assert np.isfinite(out[0][:, far]).all()
    # tiles that change path differ by rounding only
    np.testing.assert_allclose(out[0][:, far], clean[0][:, far], rtol=0, atol=1e-12 * np.abs(clean[0]).max())
