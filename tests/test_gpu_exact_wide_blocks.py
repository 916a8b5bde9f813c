"""Exact-FIRAL's gradient where the class blocks straddle one or more tiles of the product it reads
them from (64 wide in FP64, 128 in FP32): blocks wider than a tile, as wide, one off, and of one
feature.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import exact  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-9, "fp32": 1e-4}   # those of the exact path's other tests


@pytest.mark.parametrize("precision,d,c", [("fp64", 100, 3), ("fp64", 128, 2), ("fp64", 65, 4),
                                           ("fp64", 64, 3), ("fp64", 1, 130), ("fp32", 127, 4),
                                           ("fp32", 128, 3), ("fp32", 86, 5), ("fp32", 1, 260)])
def test_gradient_over_wide_blocks(precision, d, c):
    from paper_2409_07392_gb300 import api, build
    build.build()
    n = 260
    p = make_problem(n, d, c, seed=d + c)
    z = np.random.default_rng(d).gamma(2.0, 1.0, n)
    z *= 10.0 / z.sum()
    Ho, Hp = exact.h_o(p), exact.h_p(p)
    f_ref, g_ref = exact.objective(p, z, Ho, Hp), exact.gradient(p, z, Ho, Hp)
    dt = torch.float64 if precision == "fp64" else torch.float32
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(dt)
    prob = api.Problem(api.Handle(), t(p.X), t(p.h), t(p.Xo), t(p.ho), p.lam, precision=precision)
    f, g = prob.exact_objective(t(z))
    g = g.double().cpu().numpy()
    assert abs(f - f_ref) < TOL[precision] * abs(f_ref)
    assert np.linalg.norm(g - g_ref) < TOL[precision] * np.linalg.norm(g_ref)
    prob.close()
