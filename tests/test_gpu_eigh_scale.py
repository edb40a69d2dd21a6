"""Symmetric matrices at the ends of the FP32 range, tridiagonal (nothing to eliminate, so only a reflector's own entry is
squared) and full.  Bounds of tests/test_gpu_trd.py, relative to the matrix: H V = V diag(S) within 1e-5 ||H||_2
sqrt(n), V^T V = I within 1e-5."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 20, 130, 300, 1100])
@pytest.mark.parametrize("scale", [1e-25, 1e16, 1e20, 1e30])
@pytest.mark.parametrize("full", [False, True])
def test_scaled_matrices(n, scale, full):
    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(n)
    h = torch.randn(n, n, generator=g, dtype=torch.float64)
    h = (h + h.T) / 2
    if not full:
        h = torch.diag(torch.diagonal(h)) + torch.diag(torch.diagonal(h, 1), 1) + torch.diag(torch.diagonal(h, 1), -1)
    h = torch.stack([h * scale, h]).float()
    s, vt = (x.cpu().double() for x in P.eigh(h.cuda()))
    for b in range(2):
        hd, v = h[b].double(), vt[b].T
        nrm = float(torch.linalg.eigvalsh(hd).abs().max())
        assert torch.isfinite(s[b]).all() and torch.isfinite(v).all()
        assert torch.linalg.matrix_norm((hd @ v - v * s[b]) / nrm) <= 1e-5 * n ** 0.5
        assert (v.T @ v - torch.eye(n, dtype=torch.float64)).abs().max() <= 1e-5
