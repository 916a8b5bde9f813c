"""FP32 block sums over few (kind, class) rows: the diagonal part of the apply (S alone, up to 8
classes) and S with the preconditioner blocks (up to 4), on either side of that line, over one and
several row ranges, at the widths where the kernels change.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import approx  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


@pytest.mark.parametrize("c", [2, 3, 4, 5, 8, 9])
@pytest.mark.parametrize("n,d", [(300, 1), (257, 17), (5000, 50), (3001, 56), (2000, 57), (700, 64),
                                 (4001, 112), (1500, 113), (20000, 128),
                                 (16383, 20), (16500, 20)])
def test_apply_and_solve(n, d, c):
    """Elementwise on the apply: an f32 sum of L terms in any order errs by at most L 2^-24 of the
    terms' magnitudes (n + m rows, d features, c classes and 8 roundings a term).  The solve: two
    preconditioned iterations, blocks with condition below 1e3 (ridge 1e-2), so 1e-3 in norm."""
    from paper_2409_07392_gb300 import api, build
    build.build()
    lam, m = 1e-2, 2 * c
    p = make_problem(n, d, c, seed=n + c, m_o=m, x_dtype="float32", h_dtype="float32")
    p.lam = lam
    rng = np.random.default_rng(d)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    z = rng.gamma(2.0, 1.0, n)
    z = f32(z * (9.0 / z.sum()))
    V = f32(rng.standard_normal((3, d * c)))
    prob = api.Problem(api.Handle(), dev(p.X), dev(p.h), dev(p.Xo), dev(p.ho), lam,
                       precision="fp32")
    ops = approx.Operators(p)
    out = prob.hessian_apply(dev(V), dev(z)).double().cpu().numpy()
    ref = ops.sigma_apply(z, V.T).T
    X, h = np.concatenate([p.Xo, p.X]), np.concatenate([p.ho, p.h])
    w = np.concatenate([np.ones(m), z])
    Va = np.abs(V).reshape(3, c, d)
    g = np.einsum("ie,ske->isk", np.abs(X), Va)
    al = np.einsum("isk,ik->is", g, h)
    mag = np.einsum("isk,ie->ske", (g + al[:, :, None]) * (w[:, None] * h)[:, None], np.abs(X))
    mag = (mag + lam * Va).reshape(3, -1)
    assert np.all(np.abs(out - ref) <= (n + m + d + c + 8) * 2.0 ** -24 * mag)
    chol = approx.block_cholesky(ops.precond_blocks(z))
    ref = approx.pcg(lambda Y: ops.sigma_apply(z, Y), V.T, lambda R: approx.block_solve(chol, R),
                     fixed_iters=2)[0]
    got = prob.pcg(dev(z), dev(V), fixed_iters=2)[0].double().cpu().numpy().T
    assert np.linalg.norm(got - ref) <= 1e-3 * np.linalg.norm(ref)
    prob.close()
