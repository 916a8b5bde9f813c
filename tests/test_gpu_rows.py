"""The CUDA-core row contractions (FP32 and FP64 Hessian apply, quadratic forms, block sums,
Round picks) against the FP64 oracle at the edges of their tiles: class counts and feature
widths around the 4-wide groups, the 64- and 128-column tiles and the 16-feature steps, odd rows
(single-value loads), even rows (8-byte loads) and multiples of four (16-byte loads), one to
several row ranges, one to more units than a block takes.  Needs a GPU."""
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


def dev(a, dt):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().to(dt)


SHAPES = [  # n, d, c, s, labelled rows
    (1, 1, 2, 1, 0), (127, 3, 5, 1, 5), (129, 16, 4, 3, 4), (700, 17, 10, 20, 10),
    (300, 50, 10, 17, 10), (1500, 64, 33, 2, 33), (260, 65, 64, 5, 64), (515, 96, 31, 3, 0),
    (400, 97, 66, 4, 66), (333, 128, 129, 2, 129), (2100, 8, 128, 33, 128), (600, 20, 260, 3, 7),
]


def bound(p, z, A, B=None):
    """Elementwise bound of an f32 (or f64) evaluation: a sum of L terms in any order errs by at
    most L u times the sum of the terms' magnitudes; the terms are products of at most four
    rounded factors.  Magnitudes: the same expressions on absolute values with all signs plus."""
    X = np.concatenate([p.Xo, p.X])
    h = np.concatenate([p.ho, p.h])
    w = np.concatenate([np.ones(len(p.Xo)), z])
    s, D = A.shape
    V = np.abs(A).reshape(s, p.c, p.d)
    g = np.einsum("ie,ske->isk", np.abs(X), V)
    al = np.einsum("isk,ik->is", g, h)
    if B is None:
        out = np.einsum("isk,ie->ske", (g + al[:, :, None]) * (w[:, None] * h)[:, None, :],
                        np.abs(X)) + 1e-3 * V
        return out.reshape(s, D), len(X) + p.d + p.c + 8
    gb = np.einsum("ie,ske->isk", np.abs(X), np.abs(B).reshape(s, p.c, p.d))
    q = np.einsum("isk,ik->i", g * gb, h) + (al * np.einsum("isk,ik->is", gb, h)).sum(1)
    return q[len(p.Xo):] / s, 2 * p.d + p.c + s + 8


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,d,c,s,m", SHAPES)
def test_apply_forms_blocks_at_tile_edges(api, precision, n, d, c, s, m):
    f64 = precision == "fp64"
    u = 2.0 ** -52 if f64 else 2.0 ** -23
    dt = torch.float64 if f64 else torch.float32
    p = make_problem(n, d, c, seed=n + d, m_o=m, x_dtype="float64" if f64 else "float32",
                     h_dtype="float64" if f64 else "float32")
    rng = np.random.default_rng(c)
    z = rng.gamma(2.0, 1.0, n)
    z *= 7.0 / z.sum()
    A, B = rng.standard_normal((s, d * c)), rng.standard_normal((s, d * c))
    if not f64:
        z, A, B = (a.astype(np.float32).astype(np.float64) for a in (z, A, B))
    H = api.Handle()
    prob = api.Problem(H, dev(p.X, dt), dev(p.h, dt), dev(p.Xo, dt) if m else None,
                       dev(p.ho, dt) if m else None, p.lam, precision=precision)
    ops = approx.Operators(p)
    out = prob.hessian_apply(dev(A, dt), dev(z, dt)).double().cpu().numpy()
    ref = ops.sigma_apply(z, A.T).T
    mag, L = bound(p, z, A)
    assert np.all(np.abs(out - ref) <= L * u * mag)
    out = prob.hessian_apply(dev(A, dt), op=1).double().cpu().numpy()
    ref = ops.hp_apply(A.T).T
    assert np.all(np.abs(out - ref) <= L * u * bound(p, np.full(n, 1.0 / n), A)[0])
    g = prob.quad_forms(dev(A, dt), dev(B, dt)).double().cpu().numpy()
    ref = -approx.quad_forms(p.X.astype(np.float64), p.h.astype(np.float64), A.T, B.T)
    mag, L = bound(p, z, A, B)
    assert np.all(np.abs(g - ref) <= L * u * mag)
    for zz in (z, None):
        P = prob.precond_blocks(None if zz is None else dev(zz, dt)).cpu().numpy()
        w = np.concatenate([np.ones(m), np.zeros(n) if zz is None else zz])
        X, h = np.concatenate([p.Xo, p.X]), np.concatenate([p.ho, p.h]).astype(np.float64)
        q = w[:, None] * h * (1 - h)
        ref = np.einsum("ik,ie,if->kef", q, X, X) + 1e-3 * np.eye(d)
        mag = np.einsum("ik,ie,if->kef", q, np.abs(X), np.abs(X)) + 1e-3 * np.eye(d)
        assert np.all(np.abs(P - ref) <= (n + m + 8) * u * mag)
    prob.close()


@pytest.mark.parametrize("n,d,c,b", [(300, 5, 3, 3), (500, 33, 18, 3), (400, 64, 7, 2),
                                     (260, 65, 4, 2), (200, 128, 3, 2)])
def test_round_scores_at_tile_edges(api, n, d, c, b):
    """FP32 picks equal the oracle's while its top-1/top-2 gap exceeds 1e-4 (a score is a ratio
    of two sums of d^2 rounded terms: d^2 u is at most 1e-3, its square root below 1e-5)."""
    p = make_problem(n, d, c, seed=d)
    z = np.full(n, 5.0 / n)
    ref, info = approx.round_select(p, z, b, record=True)
    t = lambda a: dev(a, torch.float32)
    H = api.Handle()
    prob = api.Problem(H, t(p.X), t(p.h), t(p.Xo), t(p.ho), p.lam, precision="fp32")
    sel = prob.round(t(z), b)[0].cpu().tolist()
    prob.close()
    for k, (x, y) in enumerate(zip(sel, ref)):
        if info["gap"][k] <= 1e-4:
            break
        assert x == y, (k, sel, ref)
