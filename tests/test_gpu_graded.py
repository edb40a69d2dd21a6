"""Inputs whose rows or columns are of very different sizes (features in different units, weighted equations). The
results are compared part by part, each relative to itself: a method that keeps only the accuracy relative to the
largest entry shows in the small parts.

Bounds, derived before the first run: a column of QR errs by 4 sqrt(m) 2^-24 + 2^-19 of its norm
(test_gpu_split16.py)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


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
