"""The gradient of <G, U diag(f s) V^T> through the library's forward and backward, plain and mixed, at the default
regularization, on spectra with wide gaps and ragged sizes: against Algorithm 4 in FP64 from the oracle's factors.  The
function has no sign or rotation to fix, so no convention enters.  Bar of tests/test_gpu_bwd.py: 1e-3 relative."""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import psvd_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,n", [(40, 33), (64, 64), (130, 100), (300, 129)])
def test_gradient_of_a_spectral_function(m, n, precision):
    import paper_2609_32505_gb300 as P
    a = W.constructed(7, m, n, W.linear_spectrum(n))[0].astype(np.float32)
    gy = W.rng_for(8).standard_normal((m, n))
    f = np.linspace(1.0, 2.0, n)
    A = torch.from_numpy(a).cuda().requires_grad_(True)
    u, s, vt = P.svd(A, precision=precision)
    y = (u * (s * torch.from_numpy(f).float().cuda())[None, :]) @ vt
    (g,) = torch.autograd.grad(y, A, grad_outputs=torch.from_numpy(gy).float().cuda())
    a64 = a.astype(np.float64)
    U, S, VT, _ = O.svd(a64)
    core = U.T @ gy @ VT.T
    sf = S * f
    ref = O.svd_bwd(a64, U, S, VT, (gy @ VT.T) * sf[None, :], np.diag(core) * f, sf[:, None] * (U.T @ gy), eps=1e-8,
                    kreg_mode=0)
    g = g.cpu().double().numpy()
    assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref)
