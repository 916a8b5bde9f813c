"""Branches that the tile counts and storage types choose (needs a GPU): Round's score kernel with
one and with two point tiles per item, Round's ordered block sums on the padded tile, the stacked
rows of pooled problems, and the fused apply's (segment, probe group) items."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import approx  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_2409_07392_gb300 import api as a, build
    build.build()
    return a


@pytest.fixture(scope="module")
def handle(api):
    return api.Handle()


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# one tile per item up to 152 tiles of 128 points, two beyond; a last item of one tile, of one
# point, and full; several class chunks (c > 128) keep one tile; one chunk exactly full
@pytest.mark.parametrize("n,d,c", [(19456, 16, 5), (19457, 16, 5), (19585, 12, 7), (38912, 16, 3),
                                   (38913, 20, 4), (20000, 8, 130), (19500, 8, 128), (1, 16, 4),
                                   (129, 70, 6)])
def test_round_scores_over_item_shapes(api, handle, n, d, c):
    """First picks against the FP64 oracle where its top-1/top-2 gap exceeds 1e-3, as in the mixed
    Round tests; otherwise a near tie.  The reported point must also be unselected."""
    p = make_problem(n, d, c, seed=n % 97 + d, x_dtype="bf16", h_dtype="float32")
    b = min(3, n)
    prob = api.Problem(handle, dev(p.X).to(torch.bfloat16), dev(p.h),
                       dev(p.Xo).to(torch.bfloat16), dev(p.ho), p.lam, precision="mixed")
    z = np.full(n, float(b) / n)
    ref, info = approx.round_select(p, z, b, record=True)
    sel = prob.round(dev(z.astype(np.float32)), b)[0].cpu().tolist()
    assert len(set(sel)) == b and min(sel) >= 0 and max(sel) < n
    for t in range(b):
        if sel[t] == ref[t]:
            continue
        sc = info["scores"][t]
        assert info["gap"][t] <= 1e-3, (t, sel, ref)
        assert sc[sel[t]] >= sc[ref[t]] - 1e-3 * abs(sc[ref[t]]), (t, sc[sel[t]], sc[ref[t]])
        break


def test_round_ties_take_the_lowest_index(api, handle):
    """Equal points have equal scores, bit for bit: the first of them wins wherever the two lie
    (other tile of the item, other item, other block), although the f32 bound skips most FP64
    sums."""
    p = make_problem(25000, 16, 6, seed=5, x_dtype="bf16", h_dtype="float32")
    X, h = dev(p.X).to(torch.bfloat16), dev(p.h)
    z = torch.full((p.n,), 1.0 / p.n, dtype=torch.float32, device="cuda")

    def first():
        prob = api.Problem(handle, X, h, dev(p.Xo).to(torch.bfloat16), dev(p.ho), p.lam,
                           precision="mixed")
        s = prob.round(z, 1)[0].cpu().tolist()[0]
        prob.close()
        return s

    best = first()
    for j in (best + 128, best + 129, best + 256, 24999, 3):
        j %= p.n
        if j == best:
            continue
        keep = X[j].clone(), h[j].clone()
        X[j], h[j] = X[best], h[best]
        # the duplicate moves Sigma by one row in 25,000: the pair stays on top of the others by
        # its gap, and of the pair the lower index wins
        assert first() in (min(best, j),), (best, j)
        X[j], h[j] = keep


@pytest.mark.parametrize("d", [56, 57, 63, 64, 112, 113, 126, 128])
@pytest.mark.parametrize("n,c", [(700, 5), (5003, 9)])
def test_ordered_blocks_padded_tile(api, handle, n, c, d):
    """B_k alone (the ordered sums) on either side of the padded tiles' range: f32 sums of n terms,
    each with three roundings, against float64 (bound n 2^-24 on the terms' absolute sum)."""
    p = make_problem(n, d, c, seed=d, x_dtype="float32", h_dtype="float32")
    prob = api.Problem(handle, dev(p.X), dev(p.h), dev(p.Xo), dev(p.ho), p.lam, precision="fp32")
    g = torch.Generator(device="cuda").manual_seed(d)
    z = torch.rand(n, generator=g, device="cuda", dtype=torch.float32)
    B = prob.precond_blocks(z)
    B = (B if torch.is_tensor(B) else B[0]).double().cpu().numpy().reshape(c, d, d)
    X = np.concatenate([p.Xo, p.X]).astype(np.float32).astype(np.float64)
    h = np.concatenate([p.ho, p.h]).astype(np.float32).astype(np.float64)
    w = np.concatenate([np.ones(len(p.Xo)), z.double().cpu().numpy()])
    for k in range(c):
        a = w * h[:, k] * (1 - h[:, k])
        ref = (X * a[:, None]).T @ X + p.lam * np.eye(d)
        mag = (np.abs(X) * a[:, None]).T @ np.abs(X) + p.lam * np.eye(d)
        assert np.all(np.abs(B[k] - ref) <= (len(w) + 8) * 2.0 ** -24 * mag), k


@pytest.mark.parametrize("x_dtype,h_dtype", [("bf16", "float32"), ("float32", "float64"),
                                             ("float64", "float32")])
def test_pooled_rows_from_every_storage_type(api, handle, x_dtype, h_dtype):
    """Pools of unequal d and c, with and without labelled rows in the storage types a pool may
    have, stacked into one problem: each pool's z as accurate as the pool solved alone."""
    shapes = [(1500, 33, 6), (901, 40, 3), (2049, 64, 11), (640, 35, 17)]
    dicts = []
    for i, (n, d, c) in enumerate(shapes):
        p = make_problem(n, d, c, seed=i, x_dtype="bf16", h_dtype="float32")
        xt = {"bf16": torch.bfloat16, "float32": torch.float32, "float64": torch.float64}[x_dtype]
        ht = {"float32": torch.float32, "float64": torch.float64}[h_dtype]
        dicts.append(dict(X=dev(p.X).to(xt), h=dev(p.h).to(ht), Xo=dev(p.Xo).to(xt),
                          ho=dev(p.ho).to(ht), lam=p.lam, budget=10.0 + i))
    kw = dict(s=8, T=3, fixed_iters=5, seed=2, handle=handle)
    zs = api.batched_relax(dicts, precision="mixed", **kw)
    for dct, z in zip(dicts, zs):
        def single(prec):
            return api.relax(dct["X"], dct["h"], dct["Xo"], dct["ho"], dct["lam"], dct["budget"],
                             precision=prec, **kw)[0].double()
        z32 = single("fp32")
        e_pooled = float((z.double() - z32).norm() / z32.norm())
        e_single = float((single("mixed") - z32).norm() / z32.norm())
        assert e_pooled < 1.25 * e_single + 1e-5, (e_pooled, e_single)


@pytest.mark.parametrize("n,d,c", [(17000, 128, 4), (8500, 128, 9)])
def test_block_sums_in_several_passes(api, handle, n, d, c):
    """FP32 block sums whose operands exceed one pass (512 MiB; the second shape stays within it):
    the diagonal part S through one Hessian apply, against float64 with the sum bound (n + m + d +
    c + 8 roundings of f32 on the magnitudes)."""
    p = make_problem(n, d, c, seed=c, x_dtype="float32", h_dtype="float32")
    prob = api.Problem(handle, dev(p.X), dev(p.h), dev(p.Xo), dev(p.ho), p.lam, precision="fp32")
    g = torch.Generator(device="cuda").manual_seed(c)
    z = torch.rand(n, generator=g, device="cuda", dtype=torch.float32) / n
    V = torch.randn((2, c * d), generator=g, device="cuda", dtype=torch.float32)
    out = prob.hessian_apply(V, z).double().reshape(2, c, d)
    X = torch.cat([dev(p.Xo), dev(p.X)]).double()
    h = torch.cat([dev(p.ho), dev(p.h)]).double()
    w = torch.cat([torch.ones(len(p.Xo), device="cuda", dtype=torch.float64), z.double()])
    Vd = V.double().reshape(2, c, d)

    def form(X, V, sign):
        t = torch.einsum("ie,ske->isk", X, V)
        al = torch.einsum("isk,ik->is", t, h)
        return torch.einsum("isk,ie->ske", (t + sign * al[:, :, None]) * (w[:, None] * h)[:, None],
                            X) + p.lam * V
    ref, mag = form(X, Vd, -1.0), form(X.abs(), Vd.abs(), 1.0)
    assert bool(((out - ref).abs() <= (len(w) + d + c + 8) * 2.0 ** -23 * mag).all())
