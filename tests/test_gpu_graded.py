"""Inputs whose rows or columns are of very different sizes (features in different units, weighted equations). The
results are compared block by block, each relative to itself: a method that keeps only the accuracy relative to the
largest entry shows in the small blocks.

Bounds, derived before the first run: each split keeps 22 bits of every entry, so a product errs by about 2^-22 of
the sum of its terms, a polar factor by a few of them (1e-5, the FP32-accurate gate of the method), the gradient by
25 * 3 * 2^-22 < 2e-5 (test_gpu_split16.py); a column of QR by 4 sqrt(m) 2^-24 + 2^-19 of its norm."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _rel(x, ref):
    return np.linalg.norm(x - ref) / np.linalg.norm(ref)


def _orth(seed, m, n):
    return np.linalg.qr(np.random.default_rng(seed).standard_normal((m, n)))[0]


def _full(m, n):
    """Condition number 4, rows and columns of one size."""
    return _orth(7, m, n) @ ((_orth(8, n, n) * np.linspace(1.0, 4.0, n)) @ _orth(9, n, n).T)


@pytest.mark.parametrize("n", [24, 200, 257])
@pytest.mark.parametrize("t", [1e-3, 1e-5, 1e-7, 1e-9])
def test_polar_columns(n, t):
    """Half of the columns t times the size of the others: the columns of W, and the blocks of H."""
    import paper_2609_32505_gb300 as P
    a = _full(n, n)
    a[:, n // 2:] *= t
    a = a.astype(np.float32)
    u, s, vt = np.linalg.svd(a.astype(np.float64))
    w, h, info = P.polar(torch.from_numpy(a).cuda(), return_info=True)
    assert info[0]["status"] == 0
    w, h, w0, h0 = w.cpu().double().numpy(), h.cpu().double().numpy(), u @ vt, (vt.T * s) @ vt
    for c in (slice(0, n // 2), slice(n // 2, n)):
        assert _rel(w[:, c], w0[:, c]) <= 1e-5
        assert _rel(h[c, c], h0[c, c]) <= 1e-5


@pytest.mark.parametrize("m,n", [(400, 100), (260, 17), (700, 272)])
@pytest.mark.parametrize("t", [1e-4, 1e-6, 1e-8, 1e-12])
@pytest.mark.parametrize("preqr", [0, 1])
def test_polar_and_svd_rows(m, n, t, preqr):
    """Half of the rows t times the size of the others: W, and U diag(s) V^T, in either half."""
    import paper_2609_32505_gb300 as P
    a = _full(m, n)
    a[m // 2:] *= t
    a = a.astype(np.float32)
    g = a.astype(np.float64)
    ev, v = np.linalg.eigh(g.T @ g)
    ref = g @ ((v / np.sqrt(ev)) @ v.T)
    o = P.make_opts(preqr=preqr)
    w = P.polar(torch.from_numpy(a).cuda(), o)[0].cpu().double().numpy()
    u, s, vt = (x.cpu().double().numpy() for x in P.svd_fwd(torch.from_numpy(a).cuda(), o))
    for r in (slice(0, m // 2), slice(m // 2, m)):
        assert _rel(w[r], ref[r]) <= 1e-5
        assert _rel(((u * s) @ vt)[r], g[r]) <= 1e-5


@pytest.mark.parametrize("schedule", ["cans", "learned"])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_polar_batch_of_ranges(precision, schedule):
    """One batch with ordinary matrices between such of a wide range, every rung and the conservative rerun: the
    ordinary ones have the bits that they have in a batch of their own, the others' W is right in their small parts."""
    import paper_2609_32505_gb300 as P
    m, n = 300, 130
    a = np.stack([_full(m, n)] * 4)
    a[1, :, :50] *= 1e-8
    a[2, :, 7:90] *= 1e-6
    a[3, 200:] *= 1e-10
    A = torch.from_numpy(a.astype(np.float32)).cuda()
    kw = {"precision": precision, "max_iter": 64}
    if schedule == "learned":                     # far too high for matrices 1 and 2, which are then run again
        kw.update(schedule=P.SCHED_LEARNED, lower_bound=torch.full((4,), 0.05, device="cuda"))
    w, h, info = P.polar(A, P.make_opts(**kw), return_info=True)
    assert all(i["status"] == 0 for i in info), info
    if schedule == "learned":
        kw["lower_bound"] = kw["lower_bound"][:1]
    w0, h0 = P.polar(A[:1], P.make_opts(**kw))
    assert torch.equal(w[0], w0[0]) and torch.equal(h[0], h0[0])
    if precision:
        return
    w = w.cpu().double().numpy()
    for b, part in [(1, np.s_[:, :50]), (2, np.s_[:, 7:90]), (3, np.s_[200:])]:
        u, _, vt = np.linalg.svd(A[b].cpu().double().numpy(), full_matrices=False)
        assert _rel(w[b], u @ vt) <= 1e-5
        assert _rel(w[b][part], (u @ vt)[part]) <= 1e-5


@pytest.mark.parametrize("t", [1.0, 1e-3, 1e-6, 1e-8, 1e-12, 1e-18])
@pytest.mark.parametrize("m,n", [(200, 100), (300, 33), (700, 272)])
@pytest.mark.parametrize("grads", ["s", "all"])
def test_svd_backward_rows(m, n, t, grads):
    """The gradient of either half of the rows, by the formula of the backward in FP64 on the same inputs.  With
    `all`, dU is largest where U is smallest (1 / t), as the gradient of a function of the unweighted rows is."""
    import paper_2609_32505_gb300 as P
    s = W.linear_spectrum(n)
    a, q1, q2 = W.constructed(71, m, n, s)
    d = np.where(np.arange(m) < m // 2, 1.0, t)
    u64, s64, vt64 = np.linalg.svd(d[:, None] * a, full_matrices=False)
    gu, gs, gv = W.loss_weights(72, m, n)
    f32 = lambda x: np.ascontiguousarray(x).astype(np.float32)
    A, U, S, VT = f32(d[:, None] * a), f32(u64), f32(s64), f32(vt64)
    dU, dS, dVT = f32(gu / d[:, None]), f32(gs), f32(gv.T)
    cu = lambda x: torch.from_numpy(x).cuda()
    if grads == "s":
        da = P.svd_bwd(cu(A), cu(U), cu(S), cu(VT), None, cu(dS), None)
        dU, dVT = 0 * dU, 0 * dVT
    else:
        da = P.svd_bwd(cu(A), cu(U), cu(S), cu(VT), cu(dU), cu(dS), cu(dVT))
    da = da.cpu().double().numpy()
    A, U, S, VT, dU, dS, dVT = [x.astype(np.float64) for x in (A, U, S, VT, dU, dS, dVT)]
    eps = 1e-8
    B = U.T @ dU + VT @ dVT.T
    df = S[:, None] - S[None, :]
    K = df / (df * df + eps ** 0.5)
    Y = A @ VT.T
    D = S / (S * S + eps ** 0.5)
    E = np.diag(dS) - K * (B - B.T) / 2 - D[:, None] * (Y.T @ dU) * D[None, :]
    T = S[:, None] + S[None, :]
    X = (T / (T * T + eps ** 0.25)) * (E + E.T) / 2
    ref = (dU * D[None, :] + 2 * Y @ X) @ VT
    for r in (slice(0, m // 2), slice(m // 2, m)):
        assert _rel(da[r], ref[r]) <= 2e-5


@pytest.mark.parametrize("t", [1e-3, 1e-12])
@pytest.mark.parametrize("m,n", [(300, 40), (700, 272)])
def test_polar_backward_rows(m, n, t):
    """The same for the backward of W and H, next to a matrix of one size, whose bits do not depend on its neighbour."""
    import paper_2609_32505_gb300 as P
    g = np.random.default_rng(m)
    a = np.stack([_full(m, n)] * 2)
    d = np.where(np.arange(m) < m // 2, 1.0, t)[:, None]
    a[1] *= d
    a = a.astype(np.float32)
    dw, dh = g.standard_normal((2, m, n)), g.standard_normal((2, n, n))
    dw[1] /= d
    dw, dh = dw.astype(np.float32), dh.astype(np.float32)
    cu = lambda x: torch.from_numpy(x).cuda()
    w, h = P.polar(cu(a))
    da = P.polar_bwd(cu(a), w, h, cu(dw), cu(dh))
    assert torch.equal(da[0], P.polar_bwd(cu(a[:1]), w[:1], h[:1], cu(dw[:1]), cu(dh[:1]))[0])
    A, dW, dH, H = a[1].astype(np.float64), dw[1].astype(np.float64), dh[1].astype(np.float64), h[1].cpu().double().numpy()
    eps = 1e-8
    s, v = np.linalg.eigh(H)
    r = (v * (s / (s * s + eps ** 0.5))) @ v.T
    sym = lambda x: 0.5 * (x + x.T)
    c = sym(sym(dH) - r @ (A.T @ dW) @ r)
    tt = s[:, None] + s[None, :]
    x = v @ ((tt / (tt * tt + eps ** 0.25)) * (v.T @ c @ v)) @ v.T
    ref, da = dW @ r + 2.0 * A @ x, da[1].cpu().double().numpy()
    for rows in (slice(0, m // 2), slice(m // 2, m)):
        assert _rel(da[rows], ref[rows]) <= 2e-5


@pytest.mark.parametrize("m,n", [(300, 40), (257, 257), (2100, 130), (9000, 66)])
@pytest.mark.parametrize("low", [1e-4, 1e-12, 1e-30])
def test_qr_columns(m, n, low):
    """Columns from 1 down to `low`: Q is that of the columns brought to one size, R's columns go with them."""
    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(m + n)
    a = torch.randn(m, n, generator=g)
    d = torch.logspace(0.0, float(np.log10(low)), n, dtype=torch.float64)[torch.randperm(n, generator=g)]
    e = torch.exp2(torch.floor(torch.log2(d)))                 # powers of two: the scaled matrix is exact
    big = (a.double() * e[None, :]).float()
    q, r = P.qr(big.cuda())
    q1, r1 = P.qr(a.cuda())
    q, r, q1, r1 = (x.cpu().double() for x in (q, r, q1, r1))
    tol = 4 * m ** 0.5 * 2.0 ** -24 + 2.0 ** -19
    err = torch.linalg.vector_norm(q @ r - big.double(), dim=0) / torch.linalg.vector_norm(big.double(), dim=0)
    assert err.max() <= tol
    assert (q.T @ q - torch.eye(n, dtype=torch.float64)).abs().max() <= tol
    assert torch.equal(r, torch.triu(r)) and torch.all(torch.diagonal(r) >= 0)
    # a power of two per column changes nothing else
    assert torch.equal(q, q1) and torch.equal(r, r1 * e[None, :])


@pytest.mark.parametrize("m,n", [(300, 40), (2100, 130), (9000, 66), (17000, 33)])
@pytest.mark.parametrize("t", [1e-3, 1e-5, 1e-7, 1e-9, 1e-14])
def test_qr_rows(m, n, t):
    """The rows from m / 2 on t times the size of the others: Q R in either half, and Q against A R^-1.  In one batch
    with the matrix itself, whose bits do not depend on its neighbour."""
    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(m + n)
    a = torch.randn(2, m, n, generator=g)
    a[1, m // 2:] *= t
    q, r = P.qr(a.cuda())
    q0, r0 = P.qr(a[:1].cuda())
    assert torch.equal(q[0], q0[0]) and torch.equal(r[0], r0[0])
    q, r, a = q[1].cpu().double(), r[1].cpu().double(), a[1].double()
    ref = torch.linalg.solve_triangular(r, a, upper=True, left=False)
    tol = 4 * m ** 0.5 * 2.0 ** -24 + 2.0 ** -19
    for s in (slice(0, m // 2), slice(m // 2, m)):
        assert torch.linalg.matrix_norm(q[s] @ r - a[s]) <= tol * torch.linalg.matrix_norm(a[s])
        assert torch.linalg.matrix_norm(q[s] - ref[s]) <= 4 * tol * torch.linalg.matrix_norm(ref[s])
