"""The fused per-point apply (mixed precision, at most 32 classes, d <= 64) with more probes than
64 groups of 128 (probe, class) columns hold: hessian_apply and pcg take any s, for instance the
identity to form the dense Sigma_z.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import approx  # noqa: E402
from paper_2409_07392_gb300.synth import make_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (n, d, c, s): 32, 16 and 8 padded classes per probe; 65 groups and more, over 2 to 4 segments of
# 1,024 rows and the labelled rows' own
@pytest.mark.parametrize("n,d,c,s", [(1500, 20, 20, 264), (2100, 20, 20, 400), (1500, 64, 10, 640),
                                     (3000, 16, 8, 1032)])
def test_more_than_64_probe_groups(n, d, c, s):
    """Against the FP64 oracle within the fused kernels' 2e-5 (hi + lo operands: 2^-17 each, f32
    sums of 256 terms), and bit for bit against the same columns in calls of 64 probes: a column's
    products and the order of its sums depend on no other column."""
    from paper_2409_07392_gb300 import api, build
    build.build()
    p = make_problem(n, d, c, seed=s, x_dtype="bf16", h_dtype="float32", m_o=2 * c)
    prob = api.Problem(api.Handle(), dev(p.X).to(torch.bfloat16), dev(p.h),
                       dev(p.Xo).to(torch.bfloat16), dev(p.ho), p.lam, precision="mixed")
    rng = np.random.default_rng(s)
    z = rng.uniform(0.5, 1.5, n) * (20.0 / n)
    V = rng.standard_normal((s, d * c)).astype(np.float32)
    if s == d * c:
        V = np.eye(s, dtype=np.float32)
    Vd, zd = dev(V), dev(z.astype(np.float32))
    got = prob.hessian_apply(Vd, zd, op=0)
    ref = approx.Operators(p).sigma_apply(z, V.T.astype(np.float64)).T
    e = np.linalg.norm(got.double().cpu().numpy() - ref) / np.linalg.norm(ref)
    assert e < 2e-5, e
    X = prob.pcg(zd, Vd, fixed_iters=3)[0]
    for j in range(0, s, 64):
        part = Vd[j:j + 64].contiguous()
        assert torch.equal(got[j:j + 64], prob.hessian_apply(part, zd, op=0)), j
        assert torch.equal(X[j:j + 64], prob.pcg(zd, part, fixed_iters=3)[0]), j
    prob.close()
