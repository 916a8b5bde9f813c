"""FP32 Round scores: the forms x^T M x of eq. 14 are added over the features at double accuracy
from the f32 products M x.  Needs a GPU."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

LAM = 1e-3


def hadamard(k):
    H = np.ones((1, 1))
    while H.shape[0] < k:
        H = np.block([[H, H], [H, -H]])
    return H


def score_value(d, reps, h, z):
    """(X, expected score): rows of Hadamard signs times a power of two per feature, so every block
    is exactly diagonal, M1 and M2 are the f32 roundings of known numbers, and the products M x and
    x (M x) are exact; all rows have one score."""
    H = hadamard(1 << (d - 1).bit_length())
    scale = 2.0 ** -np.random.default_rng(d).integers(0, 5, d)
    X = np.tile(H[:, :d] * scale, (reps, 1))
    n, c, D = len(X), len(h), d * len(h)
    eta = 8.0 * np.sqrt(D)
    f32 = np.float32
    total = 0.0
    for hk in h:
        w = hk * (1.0 - hk)
        Ho = n * w * scale ** 2 + LAM              # labelled rows: the pool's rows, weight 1
        Sig = Ho + n * z * w * scale ** 2
        B = f32(1.0 / (np.sqrt(D) * Sig + eta * Ho))
        M1 = B * (f32(Sig) * B)                    # f32 products
        q1 = float(np.sum(M1.astype(np.float64) * scale ** 2))
        q2 = float(np.sum(B.astype(np.float64) * scale ** 2))
        total += w * q1 / (1.0 + eta * w * q2)
    return X, total


@pytest.mark.parametrize("d", [3, 8, 16, 50, 64, 65, 97, 128])
@pytest.mark.parametrize("n_units", [2, 3, 19])
def test_scores_are_added_in_double(d, n_units):
    """The two-float sums err by at most d^2 2^-48 (6e-11 at d = 128) of their terms, all positive;
    f32 sums of them err by 1e-8 and more."""
    from paper_2409_07392_gb300 import api, build
    build.build()
    c = n_units
    h = np.full(c, 1.0 / 32.0)
    h[0], h[1] = 0.5, 0.25
    z = 1.0 / 16.0
    reps = -(-150 // (1 << (d - 1).bit_length()))
    X, ref = score_value(d, reps, h, z)
    n = len(X)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
    hd = dev(np.tile(h, (n, 1)))
    prob = api.Problem(api.Handle(), dev(X), hd, dev(X), hd, LAM, precision="fp32")
    sel, st = prob.round(dev(np.full(n, z)), 1)
    assert sel.cpu().tolist() == [0]               # equal scores: the lowest index
    assert abs(st["score_last"] - ref) <= 1e-10 * ref, (st["score_last"], ref)
    prob.close()
