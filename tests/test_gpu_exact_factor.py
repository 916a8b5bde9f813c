"""Exact-FIRAL's factorisation in FP32 on a matrix whose Cholesky factor is a matrix of small
integers: with a correctly rounded root and divisions every step of the diagonal tile is exact, so
f and the gradient are, although each 2 x 2 block's condition number is up to 1e13.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("blocks,a0", [(20, 60), (60, 500), (60, 3900)])
def test_integer_cholesky_factor(precision, blocks, a0):
    """Class 0's block of Sigma_z is L L^T with L = [[p, 0], [a, 1]] along the diagonal, class 1's
    the identity (labelled rows 2 L[:, i] with h = (1/2, 0), no ridge, z = 0).  With the pool on
    the second feature of each block, f = sum of 1 / (4 blocks) over blocks of a unit pivot squared:
    1/4, and each gradient entry is -1 / (16 blocks).  A pivot or a quotient off by one unit in the
    last place moves its block's unit Schur complement by 2 a^2 2^-24 and more."""
    from paper_2409_07392_gb300 import api, build
    build.build()
    dt = torch.float32 if precision == "fp32" else torch.float64
    d = 2 * blocks
    L = np.zeros((d, d))
    for j in range(blocks):
        L[2 * j, 2 * j] = 2 * j + 3
        L[2 * j + 1, 2 * j] = a0 + 3 * j
        L[2 * j + 1, 2 * j + 1] = 1.0
    Xo = np.concatenate([2.0 * L.T, 2.0 * np.eye(d)])
    ho = np.zeros((2 * d, 2))
    ho[:d, 0] = ho[d:, 1] = 0.5
    X = np.eye(d)[1::2]
    h = np.tile([0.5, 0.0], (blocks, 1))
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda().to(dt)
    prob = api.Problem(api.Handle(), dev(X), dev(h), dev(Xo), dev(ho), 0.0, precision=precision)
    f, g = prob.exact_objective(dev(np.zeros(blocks)))
    assert abs(f - 0.25) <= 1e-6, f
    g = g.double().cpu().numpy() * (-16.0 * blocks)
    assert np.max(np.abs(g - 1.0)) <= 1e-6, np.max(np.abs(g - 1.0))
    prob.close()
