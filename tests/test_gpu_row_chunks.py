"""Row forms whose per-block partials exceed 256 MiB: the rows then run in chunks of whole tiles.
The gradient's quadratic forms (many probes), Round's FP32 scores (many classes) and Exact-FIRAL's
gradient (many class pairs), with rows picked on both sides of the chunks' borders, and the memory
the calls take.  Needs a GPU."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

MIB = 1 << 20


@pytest.fixture(scope="module")
def api():
    from paper_2409_07392_gb300 import api as a, build
    build.build()
    return a


def gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def rows(n, d, c, seed, dt):
    """n rows of unit features and class probabilities."""
    X = torch.randn(n, d, device="cuda", generator=gen(seed), dtype=dt)
    X /= X.norm(dim=1, keepdim=True)
    h = torch.softmax(torch.randn(n, c, device="cuda", generator=gen(seed + 1), dtype=dt), dim=1)
    return X, h


class Memory:
    """Bytes taken from the device since the start, the library's own cache emptied."""

    def __enter__(self):
        from paper_2409_07392_gb300 import _lib as L
        gc.collect()
        L.load().firal_cache_trim()
        torch.cuda.empty_cache()
        torch.cuda.synchronize()
        self.free = torch.cuda.mem_get_info()[0]
        return self

    def taken(self):
        torch.cuda.synchronize()
        return self.free - torch.cuda.mem_get_info()[0]

    def __exit__(self, *a):
        pass


# 125 (FP32) and 250 (FP64) blocks of probes: chunks of 268,416 and 134,208 rows
@pytest.mark.parametrize("precision,n", [("fp32", 700001), ("fp64", 350003)])
def test_quad_forms_in_chunks(api, precision, n):
    """g_i = -(1/s) sum_j [sum_k h a b - (sum_k h a)(sum_k h b)]: 2,000 probes' terms of order 1,
    each with at most 16 roundings, their sum's in double: 2^-24 16 (2^-53 2,000) of the terms."""
    dt = torch.float32 if precision == "fp32" else torch.float64
    d, c, s = 2, 2, 2000
    X, h = rows(n, d, c, 1, dt)
    A = torch.randn(s, d * c, device="cuda", generator=gen(5), dtype=dt)
    B = torch.randn(s, d * c, device="cuda", generator=gen(6), dtype=dt)
    H = api.Handle()
    prob = api.Problem(H, X, h, lam=1e-3, precision=precision)
    with Memory() as mem:
        g = prob.quad_forms(A, B)
        assert mem.taken() <= 256 * MIB + 64 * MIB, mem.taken() / MIB
    X, h, A, B = X.double(), h.double(), A.double(), B.double()
    u = 2.0 ** -24 if precision == "fp32" else 2.0 ** -53
    tol = 16 * u if precision == "fp32" else 2000 * u
    for r in (slice(0, 300), slice(134000, 134400), slice(268300, 268600), slice(n - 300, n)):
        a = torch.einsum("ie,ske->isk", X[r], A.view(s, c, d))
        b = torch.einsum("ie,ske->isk", X[r], B.view(s, c, d))
        hh = h[r][:, None, :]
        t1, t2, t3 = (hh * a * b).sum(2), (hh * a).sum(2), (hh * b).sum(2)
        ref = -(t1 - t2 * t3).mean(1)
        mag = ((hh * a * b).abs().sum(2) + (hh * a).abs().sum(2) * (hh * b).abs().sum(2)).mean(1)
        assert bool(((g[r].double() - ref).abs() <= tol * mag).all())
    prob.close()


def test_round_scores_in_chunks(api):
    """63 blocks of 16 classes: chunks of 532,608 rows.  Rows of norm 10 along five axes among rows
    of norm 0.1 score highest; they are the picks, wherever they lie."""
    n, d, c = 545000, 5, 1000
    X, h = rows(n, d, c, 3, torch.float32)
    X *= 0.1
    at = [17, 532607, 532608, 540000, n - 1]
    for k, i in enumerate(at):
        X[i] = 0.0
        X[i, k] = 10.0
        h[i] = 1.0 / c
    Xo, ho = rows(50, d, c, 7, torch.float32)
    prob = api.Problem(api.Handle(), X, h, Xo, ho, 1e-3, precision="fp32")
    z = torch.full((n,), 5.0 / n, device="cuda")
    z[at] = 0.0
    sel = prob.round(z, 5)[0].cpu().tolist()
    assert sorted(sel) == at, sel
    prob.close()


def test_exact_gradient_in_chunks(api):
    """516 blocks of 16 class pairs: chunks of 65,024 rows of 400,000, against FP64 (the exact path's
    1e-4); h twice, x and up to 512 MiB each of operands and partial sums, 256 MiB of the forms'."""
    n, d, c = 400000, 4, 128
    X, h = rows(n, d, c, 9, torch.float32)
    Xo, ho = rows(c, d, c, 11, torch.float32)
    z = torch.rand(n, device="cuda", generator=gen(13)) * (20.0 / n)
    H = api.Handle()
    with Memory() as mem:
        prob = api.Problem(H, X, h, Xo, ho, 1e-2, precision="fp32")
        f, g = prob.exact_objective(z)
        limit = (h.numel() + 8 * X.numel()) * 4 + (512 + 512 + 256 + 128) * MIB
        assert mem.taken() <= limit, (mem.taken() / MIB, limit / MIB)
    prob.close()
    t = lambda v: v.double()
    p64 = api.Problem(H, t(X), t(h), t(Xo), t(ho), 1e-2, precision="fp64")
    f64, g64 = p64.exact_objective(t(z))
    p64.close()
    assert abs(f - f64) <= 1e-4 * abs(f64)
    for r in (slice(0, 65024), slice(65024, 2 * 65024), slice(390144, n)):
        assert float((g[r].double() - g64[r]).norm() / g64[r].norm()) <= 1e-4
