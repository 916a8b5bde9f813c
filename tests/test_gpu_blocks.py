"""The FP64 block kernels at the edges of their register tiles (16-wide, instantiated up to 16,
32, 48, 64, 96 and 128 features): the factorisation behind the block-Jacobi preconditioner (PCG
iterates against the oracle's), and Round's nu, from the tridiagonal forms, against the oracle's
bisection over the eigenvalues.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import approx  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2409_07392_gb300 import api, build
    build.build()
    return api


def problem(api, d, c, n):
    p = make_problem(n, d, c, seed=d, x_dtype="float64", h_dtype="float64")
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return p, api.Problem(api.Handle(), t(p.X), t(p.h), t(p.Xo), t(p.ho), p.lam, precision="fp64")


@pytest.mark.parametrize("d", [1, 2, 15, 16, 17, 31, 32, 33, 48, 49, 64, 65, 95, 97, 113, 127, 128])
def test_factorisation_at_tile_edges(api, d):
    c, n, s, b = 3, 260, 2, 5.0
    p, prob = problem(api, d, c, n)
    z = np.random.default_rng(d).gamma(2.0, 1.0, n)
    z *= b / z.sum()
    B = np.random.default_rng(d + 1).standard_normal((d * c, s))
    ops = approx.Operators(p)
    chol = approx.block_cholesky(ops.precond_blocks(z))
    ref, _, _ = approx.pcg(lambda V: ops.sigma_apply(z, V), B,
                           lambda R: approx.block_solve(chol, R), fixed_iters=2)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X, _, _ = prob.pcg(t(z), t(B.T), fixed_iters=2)
    err = np.linalg.norm(X.cpu().numpy().T - ref) / np.linalg.norm(ref)
    # two iterations with a preconditioner of condition below 1e3 (ridge 1e-3, blocks of order
    # 1): each solve errs by cond d u, well below 1e-10
    assert err < 1e-10, err
    prob.close()


@pytest.mark.parametrize("d,c", [(1, 5), (2, 4), (3, 40), (16, 33), (17, 3), (32, 32), (33, 2),
                                 (64, 7), (65, 3), (90, 2)])
def test_round_nu_at_tile_edges(api, d, c):
    p, prob = problem(api, d, c, 200)
    z = np.full(200, 6.0 / 200)
    ref, info = approx.round_select(p, z, 3, record=True)
    sel, st = prob.round(torch.from_numpy(z).cuda(), 3)
    assert sel.cpu().tolist() == ref
    nu = info["nu"][-1]
    # the oracle's blocks by the same formulas, nu by bisection to 1e-15: both sides err by the
    # conditioning of the spectrum, cond u < 1e-11
    assert abs(st["nu_last"] - nu) <= 1e-9 * max(1.0, abs(nu)), (st["nu_last"], nu)
    prob.close()
