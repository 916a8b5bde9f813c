"""What the performance of this framework is measured on.

Every case is a call (or a short run of calls) that a user's program makes through the
Python binding, on the seeded Gaussian-mixture inputs of the paper's workloads.  The sizes are
those of ``synth.CONFIGS``, ``bench.py`` and the tests; ``draw`` spreads them over the same
ranges, odd sizes included.  Kinds of case:

  md         one mirror-descent update of z (Algorithm 2 lines 10-11)
  apply      Sigma_z V on a prepared problem (Lemma 1), diagonal-part block sums included
  quad       the per-point quadratic forms of the gradient (eq. 11)
  pcg        the block-Jacobi preconditioned solve Sigma_z X = B
  objective  f^(z) and its gradient by torch autograd
  step       one whole MD iteration on a prepared problem
  relax      the whole Relax call on device tensors, problem preparation included
  batched    Relax on many uneven pools in one call
  round      greedy Round picks on a prepared problem (Algorithm 3)
  exact      Exact-FIRAL's objective and gradient on dense dc x dc matrices (Algorithm 1)
  al         the active-learning loop: refit, Relax and Round, round by round
"""
import math

import torch

from paper_2409_07392_gb300 import api, autograd
from paper_2409_07392_gb300.synth import batched_problems

DEV = "cuda"
LAM = 1e-3


def listed():
    return [
        # the smallest call: one MD update of the 3,000-point pool, a few microseconds of work
        dict(name="md_3k_fp32", kind="md", n=3000, d=20, c=10, precision="fp32"),
        # the paper's small problem in FP64: a whole Relax of 20 iterations at the default
        # tolerance, where launches, host reads and FP64 latency count
        dict(name="relax_3k_fp64", kind="relax", n=3000, d=20, c=10, m=10, s=10, T=20, b=10.0,
             tol=0.1, fixed=0, precision="fp64"),
        # CIFAR-10-shaped embeddings in the binding's default precision (FP32), f32 storage, a
        # fixed number of CG iterations as in the paper's timings
        dict(name="relax_50k_fp32", kind="relax", n=50000, d=50, c=10, m=10, s=20, T=2, b=100.0,
             tol=0.1, fixed=5, precision="fp32"),
        # one FP32 Hessian apply at the ImageNet class count on a 20,000-point pool
        dict(name="apply_20k_c1000_fp32", kind="apply", n=20000, d=64, c=1000, m=1000, s=16,
             b=1000.0, precision="fp32"),
        # the CIFAR-10 shape differentiated by torch autograd, mixed precision, CG to 1e-3
        dict(name="objective_50k_mixed", kind="objective", n=50000, d=50, c=10, m=10, s=20,
             b=100.0, tol=1e-3, precision="mixed"),
        # the gradient's forms at the pipeline's feature width and class count, general operands
        dict(name="quad_200k_c100_mixed", kind="quad", n=200000, d=128, c=100, m=100, s=16,
             precision="mixed"),
        # a solve at an odd size (the Caltech-101 shape) in the default precision, 10 iterations
        dict(name="pcg_1715_c101_fp32", kind="pcg", n=1715, d=100, c=101, m=101, s=10, b=101.0,
             tol=0.1, fixed=10, precision="fp32"),
        # the headline workload: one MD iteration on the ImageNet-shaped pool of a million points
        dict(name="step_1m_c1000_fast", kind="step", n=1000000, d=64, c=1000, m=1000, s=16,
             b=1000.0, tol=0.1, fixed=10, precision="mixed_fast"),
        # 64 uneven pools in one call (preparation, one eager iteration, graph replays)
        dict(name="batched_64_mixed", kind="batched", pools=64, shapes=0, s=8, T=4, fixed=5,
             precision="mixed"),
        # four greedy picks on the full-size pipeline pool
        dict(name="round_1m_c100_mixed", kind="round", n=1000000, d=128, c=100, m=100, b=4,
             precision="mixed"),
        # Table 5's exact comparison at the ImageNet-50 shape: dense 2500 x 2500 matrices
        dict(name="exact_5k_c50_fp32", kind="exact", n=5000, d=50, c=50, m=50, b=50.0,
             precision="fp32"),
        # one round of active learning at the ImageNet-50 shape in the default precision
        dict(name="al_5k_c50_fp32", kind="al", n=5000, d=50, c=50, m=50, s=10, T=4, rounds=1,
             b=10, tol=0.1, precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a kind, then sizes over the range that kind is used in."""
    kind = rng.choice(["md", "apply", "apply", "quad", "pcg", "objective", "step", "relax",
                       "batched", "round", "exact", "al"])
    prec = rng.choice(["fp64", "fp32", "fp32", "mixed", "mixed_fast"])
    d = rng.randint(8, 128)
    s = rng.choice([4, 8, 10, 16, 20])
    if kind == "md":
        return dict(kind=kind, n=_log_int(rng, 1000, 1000000), d=16, c=8,
                    precision=rng.choice(["fp32", "fp64"]))
    if kind in ("apply", "quad", "pcg", "objective", "step", "relax"):
        if kind in ("pcg", "relax"):          # the plain precisions
            prec = rng.choice(["fp64", "fp32"])
        c = _log_int(rng, 50 if kind == "pcg" else 10, 1000)
        if kind == "step" and prec.startswith("mixed"):
            c = _log_int(rng, 300, 1000)
        if kind == "objective":               # few classes: the CIFAR-10 range
            prec, c, d = "mixed", rng.randint(5, 32), rng.randint(8, 64)
        # rows so that the pass stays well below the largest listed one
        flops = {"fp64": 2e8, "fp32": 2e10, "mixed": 4e11, "mixed_fast": 4e11}[prec]
        reps = {"apply": 1, "quad": 1, "pcg": 12, "objective": 40, "step": 24, "relax": 24}[kind]
        top = min(1000000, max(1001, int(flops * 10 / (reps * c * d * s))))
        case = dict(kind=kind, n=_log_int(rng, 1000, top), d=d, c=c, m=c, s=s, precision=prec)
        if kind != "quad":
            case["b"] = float(rng.randint(10, 500))
        if kind == "objective":
            case["tol"] = 1e-3
        if kind in ("pcg", "step", "relax"):
            case["tol"] = 0.1
            case["fixed"] = {"pcg": 10, "step": 5, "relax": 0 if prec == "fp64" else 4}[kind]
        if kind == "relax":
            case["T"] = 2
        return case
    if kind == "batched":
        return dict(kind=kind, pools=rng.randint(8, 64), shapes=rng.randint(1, 10000), s=8,
                    T=rng.randint(2, 4), fixed=rng.choice([3, 5]), precision="mixed")
    if kind == "round":
        prec = rng.choice(["fp32", "mixed"])
        c = _log_int(rng, 5, 200)
        top = min(500000, int((1e11 if prec == "mixed" else 1e10) / (c * d * d)))
        return dict(kind=kind, n=_log_int(rng, 1000, max(1001, top)), d=d, c=c, m=c,
                    b=rng.randint(2, 6), precision=prec)
    if kind == "exact":
        c, d = rng.randint(5, 50), rng.randint(10, 50)
        return dict(kind=kind, n=_log_int(rng, 500, 5000), d=d, c=c, m=c, b=float(c),
                    precision="fp32")
    c, d = rng.randint(5, 50), rng.randint(10, 64)
    return dict(kind=kind, n=_log_int(rng, 1000, 5000), d=d, c=c, m=c, s=10, T=3,
                rounds=rng.randint(1, 2), b=rng.randint(5, 10), tol=0.1, precision="fp32")


# --------------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)


def _mixture(n, d, c, m, seed, anisotropic=False):
    """(X, labels, Xo, W) in f32: one component per class, means N(0, 4 I), unit rows; the
    labelled set is one draw per component.  The anisotropic form has per-feature variances
    log-uniform in [1e-2, 1] and Zipf(1.1) priors."""
    g = _gen(seed)
    means = 2.0 * torch.randn(c, d, device=DEV, generator=g)
    W = torch.randn(c, d, device=DEV, generator=g)
    if anisotropic:
        std = torch.exp(0.5 * math.log(1e-2) * torch.rand(c, d, device=DEV, generator=g))
        prior = torch.arange(1, c + 1, device=DEV, dtype=torch.float32) ** -1.1
    else:
        std = torch.ones(c, d, device=DEV)
        prior = torch.ones(c, device=DEV)
    y = torch.multinomial(prior, n, replacement=True, generator=g)
    yo = torch.arange(m, device=DEV) % c

    def rows(lab):
        x = means[lab] + std[lab] * torch.randn(lab.numel(), d, device=DEV, generator=g)
        return x / x.norm(dim=1, keepdim=True)
    return rows(y), y, rows(yo), W


def _probs(X, W):
    """softmax(W x) in f32, in row chunks."""
    h = torch.empty(X.shape[0], W.shape[0], device=DEV, dtype=torch.float32)
    for a in range(0, X.shape[0], 1 << 17):
        h[a:a + (1 << 17)] = torch.softmax(X[a:a + (1 << 17)].float() @ W.t(), dim=1)
    return h


def _pool(case, seed):
    """The stored inputs (X, h, Xo, ho): bf16 X for the mixed precisions, else the vec type."""
    prec = case["precision"]
    X, _, Xo, W = _mixture(case["n"], case["d"], case["c"], case["m"], seed,
                           anisotropic=case["kind"] == "round")
    if prec.startswith("mixed"):
        X, Xo = X.to(torch.bfloat16), Xo.to(torch.bfloat16)
    h, ho = _probs(X, W), _probs(Xo, W)
    if prec == "fp64":
        X, Xo, h, ho = X.double(), Xo.double(), h.double(), ho.double()
    return X, h, Xo, ho


def _vdt(prec):
    return torch.float64 if prec == "fp64" else torch.float32


def _z(n, b, seed, dt):
    """A point of the budget simplex as the iterations produce it: positive, uneven."""
    z = torch.exp(0.5 * torch.randn(n, device=DEV, generator=_gen(seed + 101)))
    return (z.double() * (b / z.double().sum())).to(dt)


def _vectors(s, D, seed, dt):
    return torch.randn(s, D, device=DEV, generator=_gen(seed + 202)).to(dt)


def _signs(s, D, seed, dt):
    return (torch.randint(0, 2, (s, D), device=DEV, generator=_gen(seed + 303)) * 2 - 1).to(dt)


def _md_inputs(case, seed):
    dt = _vdt(case["precision"])
    z = _z(case["n"], 10.0, seed, dt)
    g = -torch.rand(case["n"], device=DEV, generator=_gen(seed + 404)).to(dt) - 0.01
    return z, g


def _batch(case, seed):
    out = []
    for i, sh in enumerate(batched_problems(case["pools"], seed=case["shapes"])):
        X, _, Xo, W = _mixture(sh["n"], sh["d"], sh["c"], sh["c"], seed * 1000 + i)
        X, Xo = X.to(torch.bfloat16), Xo.to(torch.bfloat16)
        out.append(dict(X=X, h=_probs(X, W), Xo=Xo, ho=_probs(Xo, W), lam=LAM,
                        budget=float(sh["b"])))
    return out


def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    st = dict(case=case, seed=seed, handle=api.Handle())
    if kind == "md":
        X, h, Xo, ho = _pool(dict(case, m=case["c"]), seed)
        st["prob"] = api.Problem(st["handle"], X, h, Xo, ho, LAM, precision=prec)
        st["z"], st["g"] = _md_inputs(case, seed)
        return st
    if kind == "batched":
        st["problems"] = _batch(case, seed)
        return st
    if kind == "al":
        X, y, Xo, _ = _mixture(case["n"], case["d"], case["c"], case["m"], seed)
        yo = torch.arange(case["m"], device=DEV) % case["c"]
        st["data"] = (X, y, Xo, yo)
        return st
    X, h, Xo, ho = _pool(case, seed)
    if kind == "relax":
        st["data"] = (X, h, Xo, ho)
        return st
    # the kinds on a prepared problem: it, not the inputs, is what the program keeps
    st["prob"] = api.Problem(st["handle"], X, h, Xo, ho, LAM, precision=prec)
    dt, D = _vdt(prec), case["d"] * case["c"]
    if kind == "quad":
        st["A"] = _signs(case["s"], D, seed, dt)
        st["B"] = _vectors(case["s"], D, seed, dt)
        return st
    st["z"] = _z(case["n"], float(case["b"]), seed, dt)
    if kind in ("apply", "pcg"):
        st["V"] = _vectors(case["s"], D, seed, dt)
    if kind == "step":
        st["opts"] = st["prob"].relax_opts(s=case["s"], T=1, tol=case["tol"],
                                           fixed_iters=case["fixed"], seed=seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "md":
        return st["prob"].md_step(st["z"], st["g"], 10.0)
    if kind == "apply":
        return st["prob"].hessian_apply(st["V"], st["z"])
    if kind == "quad":
        return st["prob"].quad_forms(st["A"], st["B"])
    if kind == "pcg":
        X, _, _ = st["prob"].pcg(st["z"], st["V"], tol=case["tol"], fixed_iters=case["fixed"])
        return X
    if kind == "objective":
        z = st["z"].detach().requires_grad_(True)
        f = autograd.firal_objective(z, st["prob"], seed=st["seed"], s=case["s"],
                                     tol=case["tol"])
        f.backward()
        return [f.detach().float(), z.grad]
    if kind == "step":
        z = st["z"].clone()
        st["prob"].relax_step(st["opts"], 0, case["b"], z, stats=False)
        return z
    if kind == "relax":
        X, h, Xo, ho = st["data"]
        z, fh = api.relax(X, h, Xo, ho, LAM, case["b"], s=case["s"], T=case["T"],
                          tol=case["tol"], fixed_iters=case["fixed"], seed=st["seed"],
                          precision=case["precision"], handle=st["handle"])
        return [z, fh]
    if kind == "batched":
        return api.batched_relax(st["problems"], s=case["s"], T=case["T"],
                                 fixed_iters=case["fixed"], seed=st["seed"],
                                 precision=case["precision"], handle=st["handle"])
    if kind == "round":
        sel, info = st["prob"].round(st["z"], case["b"])
        return [sel, info["nu_last"], info["score_last"]]
    if kind == "exact":
        f, g = st["prob"].exact_objective(st["z"])
        return [f, g]
    X, y, Xo, yo = st["data"]
    sel, W, fh = api.active_learning(X, y, Xo, yo, case["c"], case["rounds"], case["b"],
                                     precision=case["precision"], s=case["s"], T=case["T"],
                                     tol=case["tol"], seed=st["seed"], handle=st["handle"])
    return [sel, W, fh]


# --------------------------------------------------------------------------------- work
def _sizes(case):
    prec = case["precision"]
    xb = 2 if prec.startswith("mixed") else 8 if prec == "fp64" else 4
    return xb, 8 if prec == "fp64" else 4


def work(case):
    """Bytes and flops of the algorithm: inputs and outputs once; 4 n c d s per Hessian-type
    apply (two contractions), n c d (d + 1) per block sum, fixed CG iterations as given and one
    per solve in tolerance mode (the least a solve can take)."""
    kind = case["kind"]
    if kind == "md":
        vb = _sizes(case)[1]
        return {"bytes": 3.0 * case["n"] * vb, "flops": 6.0 * case["n"]}
    if kind == "batched":
        by = fl = 0.0
        ap = (2 * case["fixed"] + 2) * case["T"]
        for sh in batched_problems(case["pools"], seed=case["shapes"]):
            n, d, c = sh["n"], sh["d"], sh["c"]
            by += n * (2 * d + 4 * c + 4)
            fl += ap * 4.0 * n * c * d * case["s"] + case["T"] * 1.0 * n * c * d * (d + 1)
        return {"bytes": by, "flops": fl}
    xb, vb = _sizes(case)
    n, d, c, m = case["n"], case["d"], case["c"], case["m"]
    N = n + m
    rows = N * (d * xb + c * vb) + n * vb
    blocks = 1.0 * N * c * d * (d + 1)
    if kind == "exact":
        D = d * c
        pair = 1.0 * n * c * (c + 1) * d * (d + 1) / 2
        return {"bytes": rows + n * vb, "flops": 2 * pair + (1 / 3 + 2 / 3 + 2) * D ** 3}
    if kind == "round":
        return {"bytes": rows + 4.0 * case["b"],
                "flops": blocks + case["b"] * 2.0 * n * c * d * (d + 1)}
    if kind == "al":
        ap = 4.0 * N * c * d * case["s"]
        relax = case["T"] * (4 * ap + blocks)
        rnd = case["b"] * 2.0 * n * c * d * (d + 1)
        return {"bytes": case["rounds"] * N * d * 4.0,
                "flops": case["rounds"] * (relax + rnd + 2.0 * n * c * d)}
    s = case["s"]
    vec = 2.0 * s * c * d * vb
    ap = 4.0 * N * c * d * s
    if kind == "apply":
        return {"bytes": rows + vec, "flops": ap + blocks}
    if kind == "quad":
        return {"bytes": rows + vec, "flops": 4.0 * n * c * d * s}
    its = case.get("fixed") or 1
    if kind == "pcg":
        return {"bytes": rows + vec, "flops": its * ap + 2 * blocks}
    if kind == "objective":   # H_p V, a 2s-column solve, the gradient
        return {"bytes": rows + n * vb, "flops": (4 * its) * ap / 2 + ap + 2 * blocks + ap}
    step = (2 * its + 1) * ap + ap + 2 * blocks
    return {"bytes": rows + n * vb, "flops": step * case.get("T", 1)}


# --------------------------------------------------------------------------------- 64 bits
class _Ref:
    """The method in plain torch at 64 bits: rows labelled first, vectors (s, c, d)."""

    def __init__(self, X, h, Xo, ho):
        self.X, self.h = torch.cat([Xo, X]).double(), torch.cat([ho, h]).double()
        self.m, self.n = Xo.shape[0], X.shape[0]
        self.d, self.c = X.shape[1], h.shape[1]

    def chunks(self, s):
        step = max(256, min(1 << 16, int(1.5e8 / (s * self.c))))
        for a in range(0, self.m + self.n, step):
            yield slice(a, min(a + step, self.m + self.n))

    def sig_w(self, z):
        return torch.cat([torch.ones(self.m, device=DEV, dtype=torch.float64), z.double()])

    def p_w(self):
        w = torch.full((self.m + self.n,), 1.0 / self.n, device=DEV, dtype=torch.float64)
        w[:self.m] = 0
        return w

    def apply(self, w, V, lam=0.0):
        s = V.shape[0]
        Vf = V.reshape(s * self.c, self.d)
        out = torch.zeros_like(Vf)
        for r in self.chunks(s):
            x, h = self.X[r], self.h[r][:, None, :]
            g = (x @ Vf.t()).view(-1, s, self.c)
            al = (g * h).sum(2, keepdim=True)
            psi = (g - al) * h * w[r][:, None, None]
            out += psi.view(-1, s * self.c).t() @ x
        return out.view_as(V) + lam * V

    def blocks(self, w):
        P = torch.empty(self.c, self.d, self.d, device=DEV, dtype=torch.float64)
        q = w[:, None] * self.h * (1 - self.h)
        for k in range(self.c):
            P[k] = (self.X * q[:, k:k + 1]).t() @ self.X
        return P + LAM * torch.eye(self.d, device=DEV, dtype=torch.float64)

    def quad(self, A, B):
        s = A.shape[0]
        q = torch.zeros(self.m + self.n, device=DEV, dtype=torch.float64)
        for r in self.chunks(s):
            x, h = self.X[r], self.h[r][:, None, :]
            a = (x @ A.reshape(-1, self.d).t()).view(-1, s, self.c)
            b = (x @ B.reshape(-1, self.d).t()).view(-1, s, self.c)
            q[r] = ((h * a * b).sum(2) - (h * a).sum(2) * (h * b).sum(2)).sum(1)
        return -q[self.m:] / s

    def pcg(self, z, B, tol, fixed, maxit=100):
        w = self.sig_w(z)
        Li = torch.linalg.inv(self.blocks(w))

        def prec(R):
            return torch.einsum("kef,skf->ske", Li, R)

        def dot(a, b):
            return (a * b).sum((1, 2))
        X, R = torch.zeros_like(B), B.clone()
        Z = prec(R)
        P, rho, bn = Z.clone(), dot(R, Z), dot(B, B).sqrt()
        act = bn > 0
        if not fixed:
            act &= ~(bn <= tol * bn)
        for _ in range(fixed or maxit):
            if not bool(act.any()):
                break
            Q = self.apply(w, P, LAM)
            pq = dot(P, Q)
            act &= pq > 0
            a = torch.where(act, rho / pq, torch.zeros_like(pq))[:, None, None]
            X += a * P
            R -= a * Q
            if not fixed:
                act &= ~(dot(R, R).sqrt() <= tol * bn)
            Z = prec(R)
            new = dot(R, Z)
            P = torch.where(act[:, None, None], Z + (new / rho)[:, None, None] * P, P)
            rho = torch.where(act, new, rho)
        return X

    def probes(self, seed, t, s):
        D = self.d * self.c
        ctr = torch.arange(s * D, device=DEV, dtype=torch.int64) + t * s * D

        def wrap(v):
            return v - (1 << 64) if v >= (1 << 63) else v

        def shr(x, k):
            return (x >> k) & ((1 << (64 - k)) - 1)

        def mix(x):
            x = x + wrap(0x9E3779B97F4A7C15)
            x = (x ^ shr(x, 30)) * wrap(0xBF58476D1CE4E5B9)
            x = (x ^ shr(x, 27)) * wrap(0x94D049BB133111EB)
            return x ^ shr(x, 31)
        bits = mix(mix(ctr) ^ seed)
        return torch.where(bits < 0, -1.0, 1.0).double().view(s, self.c, self.d)

    def step(self, z, seed, t, s, b, tol, fixed):
        V = self.probes(seed, t, s)
        U = self.pcg(z, V, tol, fixed)
        HU = self.apply(self.p_w(), U)
        W = self.pcg(z, HU, tol, fixed)
        return _md(z, self.quad(V, W), b), float((V * HU).sum()) / s


def _md(z, g, b):
    z = z * torch.exp(-g / g.abs().max())
    return z * (b / z.sum())


def _cost64(case):
    """Seconds of the 64-bit form at about 0.5 TFLOP/s."""
    return work(case)["flops"] * {"objective": 12, "relax": 3}.get(case["kind"], 1) / 5e11


def exact(case, seed):
    kind = case["kind"]
    if kind in ("round", "al") or _cost64(case) > 12:
        return None
    if kind == "md":
        z, g = _md_inputs(case, seed)
        return _md(z.double(), g.double(), 10.0)
    if kind == "batched":
        out = []
        for p in _batch(case, seed):
            r = _Ref(p["X"], p["h"], p["Xo"], p["ho"])
            z = torch.full((r.n,), p["budget"] / r.n, device=DEV, dtype=torch.float64)
            for t in range(case["T"]):
                z, _ = r.step(z, seed, t, case["s"], p["budget"], 0.1, case["fixed"])
            out.append(z)
        return out
    X, h, Xo, ho = _pool(case, seed)
    r = _Ref(X, h, Xo, ho)
    dt, d, c = _vdt(case["precision"]), case["d"], case["c"]
    if kind == "quad":
        A = _signs(case["s"], d * c, seed, dt).double().view(-1, c, d)
        return r.quad(A, _vectors(case["s"], d * c, seed, dt).double().view(-1, c, d))
    if kind == "relax":
        z = torch.full((r.n,), case["b"] / r.n, device=DEV, dtype=torch.float64)
        fh = []
        for t in range(case["T"]):
            z, f = r.step(z, seed, t, case["s"], case["b"], case["tol"], case["fixed"])
            fh.append(f)
        return [z, fh]
    z = _z(case["n"], float(case["b"]), seed, dt).double()
    if kind == "exact":
        return _exact_dense(r, z)
    if kind == "step":
        return r.step(z, seed, 0, case["s"], case["b"], case["tol"], case["fixed"])[0]
    if kind == "objective":
        V = r.probes(seed, 0, case["s"])
        HV = r.apply(r.p_w(), V)
        S = r.pcg(z, torch.cat([V, HV]), case["tol"], 0, 500)
        U, Y = S[:case["s"]], S[case["s"]:]
        return [float((HV * U).sum()) / case["s"], r.quad(U, Y)]
    V = _vectors(case["s"], d * c, seed, dt).double().view(-1, c, d)
    if kind == "pcg":
        return r.pcg(z, V, case["tol"], case["fixed"]).reshape(-1, c * d)
    return r.apply(r.sig_w(z), V, LAM).reshape(-1, c * d)


def _exact_dense(r, z):
    """f = Tr(Sigma^-1 H_p) and g_i = -Tr(H_i Sigma^-1 H_p Sigma^-1) on dense matrices."""
    c, d = r.c, r.d

    def dense(w):
        M = torch.zeros(c * d, c * d, device=DEV, dtype=torch.float64)
        for a in range(0, r.X.shape[0], 2048):
            x, h, wr = r.X[a:a + 2048], r.h[a:a + 2048], w[a:a + 2048, None]
            K = (h[:, :, None] * x[:, None, :]).reshape(x.shape[0], -1)
            M -= K.t() @ (wr * K)
            for k in range(c):
                M[k * d:(k + 1) * d, k * d:(k + 1) * d] += (wr * h[:, k:k + 1] * x).t() @ x
        return M
    S = dense(r.sig_w(z)) + LAM * torch.eye(c * d, device=DEV, dtype=torch.float64)
    Si = torch.linalg.inv(S)
    M = Si @ dense(r.p_w()) @ Si
    f = torch.trace(S @ M)
    g = torch.empty(r.n, device=DEV, dtype=torch.float64)
    D = torch.stack([M[k * d:(k + 1) * d, k * d:(k + 1) * d] for k in range(c)])
    for a in range(0, r.n, 2048):
        x, h = r.X[r.m:][a:a + 2048], r.h[r.m:][a:a + 2048]
        K = (h[:, :, None] * x[:, None, :]).reshape(x.shape[0], -1)
        diag = torch.einsum("ie,kef,if->ik", x, D, x)
        g[a:a + 2048] = -((h * diag).sum(1) - ((K @ M) * K).sum(1))
    return [float(f), g]
