"""The work that a user of this library has it do, as cases to be timed and compared.

Every case goes through the package's public entry points the way a training or an analysis
program calls them.  Kinds:

  vectors     U, S and V^T of small matrices, as they come (`svd_fwd`);
  rank_layer  one layer of the differentiable rank truncation (`rank_demo.py`): SVD of the
              activations, soft truncation, reconstruction, and the gradients of the
              activations and of the rank;
  spectral    one training step with a penalty on the singular values (sum log(1 + (s/tau)^2)):
              forward, backward, the whole gradient of the matrix;
  bwd         the backward alone (`svd_bwd`) with dense gradients of U, S and V^T;
  shrink      forward use: SVD, Wiener shrinkage of the singular values, the denoised matrix;
  polar       orthogonalization of a batch of matrices with the learned lower bound;
  polar_step  polar decomposition and its backward;
  whiten      inverse square root of a covariance matrix from its eigendecomposition.

The vectors of close singular values are defined only up to (rounding error) / gap, so programs
on large matrices consume functions of the whole factorization (the gradient U f(S) V^T, the
denoised matrix U g(S) V^T, V h(S) V^T); those kinds return them whole.  The kind `vectors`, whose
singular values are far apart, returns the vectors themselves.

Sizes are those of the repository's configurations, tests and benchmark, and odd ones between.
"""
import math

import torch

import paper_2609_32505_gb300 as P
from paper_2609_32505_gb300 import train_schedule

DEV = "cuda"


def listed():
    return [
        # a handful of small matrices whose factors are used as they are: the smallest call, all
        # of it launches and latency (100 x 64 is the smoke test's matrix)
        dict(name="vectors_4x100x64", kind="vectors", batch=4, m=100, n=64, spectrum="linear", precision="fp32"),
        # one layer of the rank-selection demo at its size: 1024 tokens x 256 channels, eps = 0.1
        dict(name="rank_layer_1024x256", kind="rank_layer", batch=1, m=1024, n=256, spectrum="decay", eps=0.1),
        # the smallest workload configuration, one 256 x 256 matrix, as a training step
        dict(name="spectral_256", kind="spectral", batch=1, m=256, n=256, spectrum="loguniform", precision="fp32"),
        # the differentiation configuration: 64 matrices of 512 x 512 with singular values in
        # exact clusters of four
        dict(name="spectral_64x512", kind="spectral", batch=64, m=512, n=512, spectrum="clustered", precision="fp32"),
        # the rectangular configuration: 8 matrices of 4096 x 1024, Gaussian, mixed precision with
        # the QR preprocessing (the setting in which mixed precision keeps its results there)
        dict(name="shrink_8x4096x1024", kind="shrink", batch=8, m=4096, n=1024, spectrum="gauss",
             precision="mixed_preqr"),
        # the benchmark's matrix (4096 x 4096, condition number 10), plain FP32 path
        dict(name="spectral_4096_plain", kind="spectral", batch=1, m=4096, n=4096, spectrum="kappa10",
             precision="fp32"),
        # the benchmark's headline: the same step in mixed precision with the learned bound
        dict(name="spectral_4096_mixed", kind="spectral", batch=1, m=4096, n=4096, spectrum="kappa10",
             precision="mixed_learned"),
        # the benchmark's backward: dense gradients of U, S and V^T at 4096 x 4096
        dict(name="bwd_4096", kind="bwd", batch=1, m=4096, n=4096, spectrum="kappa10", eps=1e-8),
        # whitening of an odd number of features
        dict(name="whiten_1999", kind="whiten", batch=1, m=1999, n=1999, spectrum="kappa100"),
        # a batch of square weights orthogonalized with the learned bound (the learned-schedule
        # study's size)
        dict(name="polar_16x1024", kind="polar", batch=16, m=1024, n=1024, spectrum="kappa100",
             precision="fp32_learned"),
        # differentiable orthogonalization of ragged rectangular matrices
        dict(name="polar_step_2x1500x700", kind="polar_step", batch=2, m=1500, n=700, spectrum="kappa10", eps=1e-8),
        # the largest configuration: 4 weight-shaped matrices (14336 x 4096, power-law spectrum,
        # rounded to BF16), denoised
        dict(name="shrink_4x14336x4096", kind="shrink", batch=4, m=14336, n=4096, spectrum="power",
             precision="mixed_preqr"),
    ]


_KINDS = ["vectors", "rank_layer", "spectral", "spectral", "shrink", "shrink", "polar", "polar_step", "bwd", "whiten"]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(_KINDS)
    if kind == "vectors":
        n = _logint(rng, 16, 96)
        return dict(kind=kind, batch=_logint(rng, 1, 64), m=n + rng.randrange(0, 2 * n), n=n, spectrum="linear",
                    precision="fp32")
    if kind == "rank_layer":
        n = _logint(rng, 64, 512)
        return dict(kind=kind, batch=1, m=n * rng.randrange(1, 9) + rng.randrange(0, n), n=n, spectrum="decay",
                    eps=rng.choice([0.1, 1.0, 10.0]))
    n = _logint(rng, 200, 4096)
    batch = max(1, min(64, int(_logint(rng, 1, 64) * (512.0 / n) ** 2)))
    square = rng.random() < 0.5
    m = n if square else min(14336, int(n * math.exp(rng.uniform(0.0, math.log(4.0)))))
    if kind in ("spectral", "bwd"):
        c = dict(kind=kind, batch=batch, m=m, n=n, spectrum=rng.choice(["kappa10", "kappa100"]))
        if kind == "bwd":
            c["eps"] = 1e-8
        else:
            c["precision"] = rng.choice(["fp32", "fp32", "mixed_learned"]) if square else "fp32"
        return c
    if kind == "shrink":
        return dict(kind=kind, batch=batch, m=m, n=n, spectrum=rng.choice(["gauss", "power", "kappa10"]) if not square
                    else rng.choice(["power", "kappa10"]), precision=rng.choice(["fp32", "mixed_preqr"]))
    if kind == "polar":
        return dict(kind=kind, batch=batch, m=m, n=n, spectrum=rng.choice(["kappa10", "kappa100"]),
                    precision=rng.choice(["fp32", "fp32_learned"]))
    if kind == "polar_step":
        return dict(kind=kind, batch=batch, m=m, n=n, spectrum="kappa10", eps=1e-8)
    return dict(kind="whiten", batch=batch, m=n, n=n, spectrum=rng.choice(["kappa10", "kappa100"]))


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _orth(g, m, n):
    """m x n with orthonormal columns: the Q factor of a Gaussian matrix."""
    return torch.linalg.qr(_randn(g, m, n))[0]


def _spectrum(g, case):
    """(batch, n) singular values, descending; None for a plain Gaussian matrix."""
    B, n, kind = case["batch"], case["n"], case["spectrum"]
    i = torch.arange(n, device=DEV, dtype=torch.float32)
    t = i / max(n - 1, 1)
    if kind == "linear":
        s = 1.0 - 0.9 * t
    elif kind in ("kappa10", "kappa100"):
        s = float(kind[5:]) ** (1.0 - t)
    elif kind == "power":
        s = (i + 1.0) ** -0.7
    elif kind == "decay":
        s = 0.5 * math.sqrt(case["m"]) * torch.exp(-2.0 * t)
    elif kind == "loguniform":
        s = torch.exp(torch.rand(B, n, generator=g, device=DEV) * math.log(1e-3))
        return s.sort(dim=1, descending=True)[0]
    elif kind == "clustered":                     # clusters of 4 exactly equal values in [1e-2, 1]
        k = -(-n // 4)
        jit = torch.rand(B, k, generator=g, device=DEV) * 0.8 + 0.1
        c = torch.exp(math.log(1e-2) * (torch.arange(k, device=DEV) + jit) / k)
        return c.repeat_interleave(4, dim=1)[:, :n].contiguous()
    else:
        return None
    return s[None, :].expand(B, n).contiguous()


def _matrix(g, case):
    """(batch, m, n) FP32 inputs with the case's spectrum, and the factors they were made from."""
    B, m, n = case["batch"], case["m"], case["n"]
    s = _spectrum(g, case)
    if s is None:                                 # iid N(0, 1/n)
        return _randn(g, B, m, n) / math.sqrt(n), None
    a = torch.empty(B, m, n, device=DEV)
    us, vs = [], []
    for b in range(B):
        if case["spectrum"] == "power":           # weight-shaped: a scaled Gaussian left factor, BF16 values
            u = _randn(g, m, n) / math.sqrt(m)
        else:
            u = _orth(g, m, n)
        v = _orth(g, n, n)
        torch.matmul(u * s[b], v.T, out=a[b])
        if case["kind"] == "bwd":
            us.append(u)
            vs.append(v.T)
    if case["spectrum"] == "power":
        a = a.to(torch.bfloat16).float()
    if case["kind"] == "bwd":
        return a, (torch.stack(us).contiguous(), s, torch.stack(vs).contiguous())
    return a, None


def _tau(a):
    """Scale of the spectral functions: the root mean square singular value."""
    return float(torch.linalg.vector_norm(a[0]) / math.sqrt(a.shape[2]))


def prepare(case, seed):
    g = _gen(seed)
    B, m, n = case["batch"], case["m"], case["n"]
    st = {"case": dict(case)}
    if case["kind"] == "whiten":
        h = torch.empty(B, n, n, device=DEV)
        s = _spectrum(g, case)
        for b in range(B):
            q = _orth(g, n, n)
            h[b] = (q * s[b]) @ q.T
        st["a"] = 0.5 * (h + h.transpose(1, 2))
        return st
    a, fac = _matrix(g, case)
    st["a"] = a
    if case["kind"] in ("spectral", "shrink"):
        st["tau"] = _tau(a)
    if case["kind"] == "bwd":
        st["u"], st["s"], st["vt"] = fac
        st["du"], st["ds"], st["dvt"] = _randn(g, B, m, n), _randn(g, B, n), _randn(g, B, n, n)
    if case["kind"] == "rank_layer":
        st["a"] = a[0].contiguous()
        st["gy"] = _randn(g, m, n) + st["a"]       # correlated with the activations, as a reconstruction loss's is
        st["gamma"] = torch.tensor(0.35 * n, device=DEV)
    if case["kind"] == "polar_step":
        st["dw"], st["dh"] = _randn(g, B, m, n), _randn(g, B, n, n)
    if case.get("precision", "").endswith("_learned"):
        st["params"], st["margin"], probes = train_schedule.load(device=DEV)
        st["z"] = P.rademacher_probes(B, n, probes, seed=seed, device=DEV)
    return st


# ---------------------------------------------------------------- passes
def _opts(st):
    """Options of the case's precision as `svd` and `make_opts` take them."""
    p = st["case"].get("precision", "fp32")
    if p == "fp32":
        return dict(precision=P.PREC_FP32)
    if p == "mixed_preqr":
        return dict(precision=P.PREC_MIXED, preqr=1)
    lb = P.predict_lower_bound(st["a"], st["params"], st["margin"], z=st["z"])
    return dict(precision=P.PREC_MIXED if p == "mixed_learned" else P.PREC_FP32, schedule=P.SCHED_LEARNED,
                lower_bound=lb)


def run(st):
    case, a = st["case"], st["a"]
    kind = case["kind"]
    if kind == "vectors":
        u, s, vt = P.svd_fwd(a, P.make_opts(**_opts(st)))
        return {"u": u, "s": s, "vt": vt}
    if kind == "rank_layer":
        x = a.detach().requires_grad_(True)
        gamma = st["gamma"].detach().requires_grad_(True)
        u, s, vt = P.svd(x, eps=case["eps"])
        j = torch.arange(case["n"], device=DEV, dtype=torch.float32)
        y = (u * (s * torch.sigmoid((gamma - j) / 2.0))[None, :]) @ vt
        dx, dgamma = torch.autograd.grad(y, (x, gamma), grad_outputs=st["gy"])
        return {"y": y, "s": s, "dx": dx, "dgamma": dgamma}
    if kind == "spectral":
        x = a.detach().requires_grad_(True)
        _, s, _ = P.svd(x, **_opts(st))
        loss = torch.log1p((s / st["tau"]) ** 2).sum()
        (dx,) = torch.autograd.grad(loss, x)
        return {"s": s, "dx": dx}
    if kind == "bwd":
        return P.svd_bwd(a, st["u"], st["s"], st["vt"], st["du"], st["ds"], st["dvt"], eps=case["eps"])
    if kind == "shrink":
        o = _opts(st)
        u, s, vt = P.svd_fwd(a, P.make_opts(**o))
        s2 = s * s
        f = s * s2 / (s2 + st["tau"] ** 2)
        y = P.gemm_tn(u * f[:, None, :], vt.transpose(1, 2))
        return {"s": s, "y": y}
    if kind == "polar":
        o = _opts(st)
        w, h = P.polar(a, P.make_opts(**o))
        return {"w": w, "h": h}
    if kind == "polar_step":
        w, h = P.polar(a)
        return {"w": w, "h": h, "da": P.polar_bwd(a, w, h, st["dw"], st["dh"], eps=case["eps"])}
    s, vt = P.eigh(a)
    v = vt.transpose(1, 2)
    return {"s": s, "r": P.gemm_tn(v * torch.rsqrt(s)[:, None, :], v)}


# ---------------------------------------------------------------- cost and exact values
def work(case):
    """Bytes of the inputs and outputs, and operations of the standard dense algorithms: thin SVD
    with vectors 6 m n^2 + 20 n^3, symmetric eigendecomposition 9 n^3, polar decomposition through
    one SVD-free product chain 6 m n^2 + 2 n^3, each backward its products."""
    B, m, n = case["batch"], case["m"], case["n"]
    kind = case["kind"]
    mn, nn = float(m) * n, float(n) * n
    svd, bwd = 6.0 * mn * n + 20.0 * nn * n, 10.0 * mn * n + 2.0 * nn * n
    by, fl = {
        "vectors": (2 * mn + nn + n, svd),
        "rank_layer": (4 * mn + n, svd + bwd + 6.0 * mn * n),
        "spectral": (2 * mn + n, svd + 2.0 * mn * n),
        "bwd": (4 * mn + 2 * nn + 2 * n, bwd),
        "shrink": (2 * mn + n, svd + 2.0 * mn * n),
        "polar": (2 * mn + nn, 6.0 * mn * n + 2.0 * nn * n),
        "polar_step": (4 * mn + 2 * nn, 16.0 * mn * n + 15.0 * nn * n),
        "whiten": (2 * nn + n, 11.0 * nn * n),
    }[kind]
    return {"bytes": 4.0 * B * by, "flops": B * fl}


def _sym(x):
    return 0.5 * (x + x.transpose(-1, -2))


def _sigma(a64):
    """Singular values in 64 bits, descending, from the eigenvalues of A^T A (condition numbers
    here stay below 1e3, so squaring costs nothing that 32 bits could see)."""
    n = a64.shape[-1]
    if n > 2048:
        return None
    ev = torch.linalg.eigvalsh(a64.transpose(-1, -2) @ a64)
    return ev.clamp_min(0).sqrt().flip(-1)


def _exact_bwd(a, u, s, vt, du, ds, dvt, eps):
    """Algorithm 4 in 64 bits from the given factors."""
    v = vt.transpose(-1, -2)
    w, wb = u @ vt, du @ vt
    vb = dvt.transpose(-1, -2) + w.transpose(-1, -2) @ du
    p = vt @ vb
    b = 0.5 * (p - p.transpose(-1, -2))
    d = s[..., :, None] - s[..., None, :]
    k = d / (d * d + eps ** 0.5)
    hb = v @ (torch.diag_embed(ds) + k.transpose(-1, -2) * b) @ vt
    r = (v * (s / (s * s + eps ** 0.5))[..., None, :]) @ vt
    c = _sym(hb - r @ a.transpose(-1, -2) @ wb @ r)
    t = s[..., :, None] + s[..., None, :]
    x = v @ ((t / (t * t + eps ** 0.25)) * (vt @ c @ v)) @ vt
    return wb @ r + 2.0 * a @ x


def exact(case, seed):
    st = prepare(case, seed)
    kind = case["kind"]
    a = st["a"].double()
    if kind == "bwd":
        return _exact_bwd(a, *(st[k].double() for k in ("u", "s", "vt", "du", "ds", "dvt")), case["eps"])
    if kind == "vectors":
        u, s, vt = torch.linalg.svd(a, full_matrices=False)
        at = vt.abs().argmax(dim=-1, keepdim=True)
        sg = torch.sign(torch.gather(vt, -1, at))
        return {"u": u * sg.transpose(-1, -2), "s": s, "vt": vt * sg}
    if kind == "rank_layer":
        u, s, vt = torch.linalg.svd(a, full_matrices=False)
        j = torch.arange(case["n"], device=DEV, dtype=torch.float64)
        mask = torch.sigmoid((st["gamma"].double() - j) / 2.0)
        gy = st["gy"].double()
        f = s * mask
        core = u.T @ gy @ vt.T
        dx = _exact_bwd(a, u, s, vt, (gy @ vt.T) * f, torch.diagonal(core) * mask, f[:, None] * (u.T @ gy),
                        case["eps"])
        return {"y": (u * f) @ vt, "s": s, "dx": dx,
                "dgamma": (torch.diagonal(core) * s * mask * (1.0 - mask) / 2.0).sum()}
    n = case["n"]
    eye = torch.eye(n, dtype=torch.float64, device=DEV)
    if kind in ("spectral", "shrink"):
        g = a.transpose(1, 2) @ a
        c = torch.linalg.cholesky(g + st["tau"] ** 2 * eye)
        if kind == "spectral":
            # Algorithm 4 with a gradient of S alone: A (V diag(2 T_ii ds_i) V^T), T_ii = 2 s / (4 s^2 + eps^(1/4)),
            # ds = 2 s / (s^2 + tau^2), which is A times a function of A^T A (eps = 1e-8, the default of `svd`)
            reg = torch.linalg.cholesky(4.0 * g + 1e-8 ** 0.25 * eye)
            return {"s": _sigma(a), "dx": 8.0 * a @ torch.cholesky_solve(torch.cholesky_solve(g, reg), c)}
        return {"s": _sigma(a), "y": a @ torch.cholesky_solve(g, c)}
    if case["batch"] * float(n) ** 3 > 2e10:      # the eigendecompositions below would take too long
        return None
    if kind == "whiten":
        s, v = torch.linalg.eigh(a)
        return {"s": s.flip(-1), "r": (v * s.rsqrt()[:, None, :]) @ v.transpose(1, 2)}
    ev, v = torch.linalg.eigh(a.transpose(1, 2) @ a)
    s = ev.clamp_min(0).sqrt()
    vt = v.transpose(1, 2)
    h = (v * s[:, None, :]) @ vt
    w = a @ ((v / s[:, None, :]) @ vt)
    if kind == "polar":
        return {"w": w, "h": h}
    # Algorithm 3 in 64 bits
    eps, dw, dh = case["eps"], st["dw"].double(), st["dh"].double()
    r = (v * (s / (s * s + eps ** 0.5))[:, None, :]) @ vt
    b = _sym(_sym(dh) - r @ a.transpose(1, 2) @ dw @ r)
    t = s[:, :, None] + s[:, None, :]
    x = v @ ((t / (t * t + eps ** 0.25)) * (vt @ b @ v)) @ vt
    return {"w": w, "h": h, "da": dw @ r + 2.0 * a @ x}
