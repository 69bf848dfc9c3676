"""The fixed-point reconstructions keep the digits of small values and of uniform states: each stencil is
evaluated relative to its own values, whatever else its tile holds.

Flows with fronts in both directions on grids that take the path.  A transverse momentum 10^-6 and
10^-10 of the streamwise one: its flux in the sweep along the stream (no pressure in it) against the oracle at
the flux bound of test_gpu_parity.py, relative to its own largest value.  A uniform gas of low
density and pressure around a dense block: away from the block every face has the same flux, so the
residual there is zero to the bit, across tiles that the block reaches and tiles that it does not.
And Riemann data and a smooth field with random strengths on larger grids, ragged and thin, against
the oracle at the bounds of test_gpu_parity.py."""
import numpy as np
import pytest

from paper_2410_05489_gb300 import problems as P
from test_gpu_fixed import data
from test_gpu_parity import A, TOL_F, check_residual, comp_err, gpu_residual  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [1e-6, 1e-10])
@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_small_transverse_momentum(A, oracle, order, along, small):  # noqa: F811
    nx, ny = 272, 260
    pb = P.Problem(ndim=2, nx=nx, ny=ny, order=order)
    x, y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    q = (x >= 0.53).astype(int) + 2 * (y >= 0.47)
    rho, u, p = (np.array(v)[q] for v in ([1.0, 0.7, 0.5, 1.3], [0.6, 1.1, 0.9, 0.7], [1.0, 0.6, 0.4, 1.5]))
    v = small * u * (1.0 + 0.1 * np.sin(6.0 * x + 2.0) * np.sin(5.0 * y + 1.0))
    if along == "y":
        u, v = v, u
    W = P.conservative((rho, u, v, p), pb.gamma, 2)
    sx, sy = oracle.prime_sigma(pb, W)
    assert min(sx.max(), sy.max()) > pb.sigma_thres / 16.0  # fronts in both directions
    _, _, _, Fxc, Fyc, _ = oracle.residual(pb, W, sx, sy)
    _, _, _, Fx, Fy, _ = gpu_residual(A, pb, W, sx, sy)
    g, c = (Fx[2], Fxc[2]) if along == "x" else (Fy[1], Fyc[1])
    assert np.abs(c).max() < 10.0 * small
    assert comp_err(g[None], c[None]) <= TOL_F


@pytest.mark.parametrize("shape", [(900, 190), (85, 2000), (410, 402)])
@pytest.mark.parametrize("kind", ["riemann", "smooth"])
@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_residual_parity_on_larger_grids(A, oracle, order, kind, shape):  # noqa: F811
    pb, W = data(kind, shape[0], shape[1], order, 5 * order + shape[0])
    sx, sy = oracle.prime_sigma(pb, W) if kind == "riemann" else P.random_sigma(pb, order, 1.0)
    assert min(sx.max(), sy.max()) > pb.sigma_thres / 16.0
    check_residual(A, oracle, pb, W, sx, sy)


@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_uniform_gas_beside_a_front(A, order):  # noqa: F811
    import torch

    n = 300
    pb = P.Problem(ndim=2, nx=n, ny=n, order=order)
    lo, hi = (0.137, 0.31, -0.23, 0.11), (1.0, 0.5, 0.4, 1.0)
    prim = [np.full((n, n), a) for a in lo]
    for f, a in zip(prim, hi):
        f[120:170, 90:160] = a
    W = torch.as_tensor(P.conservative(prim, pb.gamma, 2), device="cuda")
    s = A.Solver(pb)
    try:
        s.W.copy_(W)
        s.prime()
        lim = pb.sigma_thres / 16.0
        assert float(s.sx.max()) > lim and float(s.sy.max()) > lim
        L, _, _ = s.residual()
    finally:
        s.close()
    far = np.ones((n, n), bool)
    far[120 - order:170 + order, 90 - order:160 + order] = False
    assert np.all(L.cpu().numpy()[:, far] == 0.0)

@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_tiles_and_launches_do_not_change_the_bits(A, order):  # noqa: F811
    """Batched (8 x 64 and 8 x 32 tiles) and alone (the planned tiles): the same strengths and states."""
    from paper_2410_05489_gb300 import batch

    shapes = [(64, 64), (100, 90), (128, 128), (150, 141), (210, 200), (300, 270)]
    probs = [P.riemann_2d(m, order, 3 * order + m, ny=k) for m, k in shapes]
    out = []
    for lines in (64, 32):
        bt = batch.Batch([p for p, _ in probs], [w for _, w in probs])
        try:
            bt.set_tiles((lines,) * 4)
            bt.run(2)
            out.append([(bt.state(i), *bt.sigma(i)) for i in range(len(probs))])
        finally:
            bt.close()
    for i, (pb, W) in enumerate(probs):
        s = A.Solver(pb, W)
        try:
            s.step()
            s.step()
            alone = [t.cpu().numpy() for t in (s.W, s.sx, s.sy)]
        finally:
            s.close()
        for a, b, c in zip(out[0][i], out[1][i], alone):
            assert np.array_equal(a, b)
            assert np.array_equal(a, c), (shapes[i], np.abs(a - c).max())
