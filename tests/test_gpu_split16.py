"""Split-FP16 products (PREC_F16X3) and the 16-column epilogues of the product kernel, through the calls
that use them, at the sizes where they change path: ragged 128 x 256 tiles, column counts off the
16-column pieces, rows off the 32-byte alignment, one k-block and a remainder; and inputs at the ends of
the FP32 range, whose powers of two must come back out of the products.

Bounds: the FP32-accurate gate of the method, 1e-5 relative in the 2-norm over the entries, for every
quantity of a matrix with condition number 10 (each split keeps 22 bits, so a product errs by about
2^-22 and a polar factor by a few of them)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _rel(x, ref):
    return np.linalg.norm(x - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("m,n", [(1, 1), (17, 3), (64, 16), (100, 15), (129, 64), (160, 129), (257, 255), (300, 257),
                                 (520, 272), (700, 400)])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e25])
def test_polar_edges_and_ranges(m, n, scale):
    import paper_2609_32505_gb300 as P
    a = np.stack([W.constructed(50 + b, m, n, W.kappa_spectrum(n, 10.0) if n > 1 else np.ones(1))[0]
                  for b in range(2)])
    a = (a * scale).astype(np.float32)
    w, h = P.polar(torch.from_numpy(a).cuda())
    w, h = w.cpu().double().numpy(), h.cpu().double().numpy()
    for b in range(2):
        u, s, vt = np.linalg.svd(a[b].astype(np.float64), full_matrices=False)
        assert _rel(w[b], u @ vt) <= 1e-5
        assert _rel(h[b], (vt.T * s) @ vt) <= 1e-5


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", [(40, 33), (130, 100), (300, 257)])
def test_svd_reconstruction_and_gradient(m, n, precision):
    # U = W V and the backward's products against FP64 on a spectrum with wide gaps
    import paper_2609_32505_gb300 as P
    a = W.constructed(7, m, n, W.linear_spectrum(n))[0].astype(np.float32)
    A = torch.from_numpy(a).cuda().requires_grad_(True)
    u, s, vt = P.svd(A, precision=precision)
    f = torch.linspace(1.0, 2.0, n, device="cuda")
    y = (u * (s * f)[None, :]) @ vt
    rec = ((u * s[None, :]) @ vt).detach().cpu().double().numpy()
    assert _rel(rec, a.astype(np.float64)) <= 1e-5
    U, S, VT = np.linalg.svd(a.astype(np.float64), full_matrices=False)
    assert _rel(y.detach().cpu().double().numpy(), (U * (S * f.cpu().double().numpy())) @ VT) <= 1e-5


@pytest.mark.parametrize("M,N,K", [(33, 16, 64), (128, 264, 65), (40, 24, 31), (257, 40, 200)])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_product_rows_off_alignment(M, N, K, precision):
    # contiguous outputs whose rows are and are not multiples of 32 bytes, at an aligned and an
    # unaligned base (the second matrix of a batch of odd sizes)
    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(M + N)
    for batch in (1, 3):
        a, b = torch.randn(batch, M, K, generator=g), torch.randn(batch, N, K, generator=g)
        d = P.gemm_tn(a.cuda(), b.cuda(), precision).cpu().double()
        ref = a.double() @ b.double().transpose(1, 2)
        tol = {0: 2.0 ** -8, 1: 2.0 ** -10, 2: 2.0 ** -19}[precision]   # operand rounding, with a factor 2
        bound = (a.double().abs() @ b.double().abs().transpose(1, 2))
        assert ((d - ref).abs() <= tol * bound + 1e-30).all()


@pytest.mark.parametrize("m,n", [(1, 1), (40, 7), (70, 33), (129, 64), (300, 257)])
@pytest.mark.parametrize("sa,su,sv,sg", [(1.0, 1.0, 1.0, 1.0), (1e6, 1.0, 1.0, 1e-12), (1e-6, 1.0, 1.0, 1e12),
                                         (1.0, 1e3, 24.0, 1.0)])
def test_backward_edges_and_ranges(m, n, sa, su, sv, sg):
    """The formula of the backward in FP64 on the same FP32 inputs, also with inputs far from 1 and with factors
    that are not orthonormal.  Bound: a product errs by about 3 * 2^-22 of the size of its terms, and the
    divided differences of an evenly spaced spectrum raise the largest term over the mean by less than 25:
    25 * 3 * 2^-22 < 2e-5."""
    import paper_2609_32505_gb300 as P
    s = W.linear_spectrum(n) if n > 1 else np.ones(1)
    a, q1, q2 = W.constructed(61, m, n, s)
    gu, gs, gv = W.loss_weights(62, m, n)
    f32 = lambda x: np.ascontiguousarray(x).astype(np.float32)
    A, U, S, VT = f32(sa * a), f32(su * q1), f32(sa * s), f32(sv * q2.T)
    dU, dS, dVT = f32(sg * gu), f32(sg / sa * gs), f32(sg * gv.T)
    t = lambda x: torch.from_numpy(x).cuda()
    da = P.svd_bwd(t(A), t(U), t(S), t(VT), t(dU), t(dS), t(dVT), 0.0, 2).cpu().double().numpy()
    A, U, S, VT, dU, dS, dVT = [x.astype(np.float64) for x in (A, U, S, VT, dU, dS, dVT)]
    B = U.T @ dU + VT @ dVT.T
    d = S[:, None] - S[None, :]
    K = np.divide(1.0, d, out=np.zeros_like(d), where=np.abs(d) > 1e-6 * S.max())
    Y = A @ VT.T
    D = 1.0 / S
    E = np.diag(dS) - K * (B - B.T) / 2 - D[:, None] * (Y.T @ dU) * D[None, :]
    X = (E + E.T) / 2 / (S[:, None] + S[None, :])
    ref = (dU * D[None, :] + 2 * Y @ X) @ VT
    assert _rel(da, ref) <= 2e-5


@pytest.mark.parametrize("m,n", [(1, 1), (3, 2), (33, 17), (65, 64), (255, 63), (257, 65), (260, 130), (513, 70),
                                 (2048, 66), (2049, 66), (2300, 40), (4100, 33), (8192, 65), (8193, 65), (16385, 33),
                                 (23024, 34)])
def test_qr_panel_shapes(m, n):
    """The panel's launch shapes: one to sixteen CTAs per matrix, 256, 512, 1024 and 1536 rows each, panels of 64 and
    32 columns, with remainders in rows and columns; the last matrix has dependent columns (a zero
    reflector).  The rounding errors of a column of m entries add up to about sqrt(m) 2^-24, those of the split
    products to a few 2^-22: 4 sqrt(m) 2^-24 + 2^-19."""
    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(m + n)
    a = torch.randn(2, m, n, generator=g)
    a[1, :, n // 2:] = 0.0
    q, r = P.qr(a.cuda())
    a, q, r = a.double(), q.cpu().double(), r.cpu().double()
    tol = 4 * m ** 0.5 * 2.0 ** -24 + 2.0 ** -19
    for b in range(2):
        assert torch.linalg.matrix_norm(q[b] @ r[b] - a[b]) <= tol * torch.linalg.matrix_norm(a[b])
        assert (q[b].T @ q[b] - torch.eye(n, dtype=torch.float64)).abs().max() <= tol
        assert torch.equal(r[b], torch.triu(r[b])) and torch.all(torch.diagonal(r[b]) >= 0)
