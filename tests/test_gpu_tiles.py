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
