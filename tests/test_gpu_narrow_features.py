"""FP64 at one to four features and many (probe, class) or (kind, class) rows: the tile of the row
contractions is then bounded by shared memory, not by threads.  Apply, solve and preconditioner
blocks against the FP64 oracle.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import approx  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float64)).cuda()


# s c = 1,000 rows in one tile; 2 x 1,000 and 2 x 500 rows of the block sums; more rows than one
# tile; few classes, where the rows' factors take the memory
@pytest.mark.parametrize("d,c,s", [(1, 100, 10), (2, 100, 10), (1, 50, 20), (2, 50, 20),
                                   (1, 1000, 2), (2, 1000, 1), (1, 500, 2), (2, 300, 9),
                                   (1, 4, 256), (2, 2, 400), (2, 6, 128), (3, 2, 600),
                                   (4, 2, 513)])
def test_fp64_narrow_features(d, c, s):
    """A double sum of L terms in any order errs by at most L 2^-53 times the terms' magnitudes:
    below 1e-12 of the result's norm for 300 rows, probes of order 1 and h below 1 (the apply's
    terms cancel by less than two digits); the solve takes two iterations at a condition below
    1e4, so 1e-8 holds with room."""
    from paper_2409_07392_gb300 import api, build
    build.build()
    n = 290
    p = make_problem(n, d, c, seed=d + c, m_o=10, x_dtype="float64", h_dtype="float64")
    prob = api.Problem(api.Handle(), dev(p.X), dev(p.h), dev(p.Xo), dev(p.ho), p.lam,
                       precision="fp64")
    rng = np.random.default_rng(s)
    z = rng.gamma(2.0, 1.0, n)
    z *= 7.0 / z.sum()
    V = rng.standard_normal((s, d * c))
    ops = approx.Operators(p)
    rel = lambda a, b: np.linalg.norm(a - b) / np.linalg.norm(b)
    out = prob.hessian_apply(dev(V), dev(z)).cpu().numpy()
    assert rel(out, ops.sigma_apply(z, V.T).T) < 1e-11
    for zz in (z, None):
        P = prob.precond_blocks(None if zz is None else dev(zz)).cpu().numpy()
        ref = ops.ho_blocks() if zz is None else ops.precond_blocks(z)
        assert rel(P, ref) < 1e-11
    chol = approx.block_cholesky(ops.precond_blocks(z))
    ref = approx.pcg(lambda Y: ops.sigma_apply(z, Y), V.T, lambda R: approx.block_solve(chol, R),
                     fixed_iters=2)[0]
    X = prob.pcg(dev(z), dev(V), fixed_iters=2)[0].cpu().numpy()
    assert rel(X.T, ref) < 1e-8
    prob.close()
