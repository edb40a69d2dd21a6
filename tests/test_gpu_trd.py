"""The on-chip tridiagonalization (csrc/trd.cu) through psvd_eigh, at the sizes where its launch shape
changes: the ends of each column width (32 .. 512 threads, one or two chunks), phases of one or two
columns more than a power of two, more matrices than fit the device at once, the first size that
the L2-streaming kernel takes over (4097), and matrices whose reflectors vanish.

H V = V diag(S) and V^T V = I with the bounds of tests/test_gpu_eigh.py (1e-5 ||H||_2 sqrt(n) and 1e-5,
the size of FP32 Householder reduction's backward error with its constant), in FP64 on the device."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _check(h):
    import paper_2609_32505_gb300 as P
    s, vt = P.eigh(h)
    torch.cuda.synchronize()
    n = h.shape[-1]
    for b in range(min(h.shape[0], 8)):
        hd, v, sd = h[b].double(), vt[b].double().T, s[b].double()
        nrm = max(float(sd.abs().max()), 1e-30)
        assert torch.linalg.matrix_norm(hd @ v - v * sd) <= 1e-5 * nrm * n ** 0.5
        assert (v.T @ v - torch.eye(n, dtype=torch.float64, device=v.device)).abs().max() <= 1e-5
        assert torch.all(sd[1:] <= sd[:-1])


def _sym(seed, batch, n):
    g = torch.Generator()
    g.manual_seed(seed)
    a = torch.randn(batch, n, n, generator=g)
    return ((a + a.transpose(1, 2)) * 0.5).cuda()


@pytest.mark.parametrize("n", [3, 4, 5, 31, 32, 33, 127, 128, 129, 130, 255, 256, 257, 511, 512, 513, 1023, 1024,
                               1025, 1027, 2047, 2048, 2049, 2051, 4095, 4096, 4097])
def test_sizes_at_the_edges_of_the_launch_shapes(n):
    _check(_sym(n, 1, n))


@pytest.mark.parametrize("batch,n", [(700, 40), (70, 300), (9, 1025), (3, 2050)])
def test_more_matrices_than_run_at_once(batch, n):
    h = _sym(batch, batch, n)
    _check(h)
    import paper_2609_32505_gb300 as P
    s, vt = P.eigh(h)
    s1, vt1 = P.eigh(h[-1:])                      # the last matrix, alone on the device
    w = torch.linalg.eigvalsh(h[-1].double()).flip(-1)
    tol = 2e-6 * float(w.abs().max()) * max(1.0, n ** 0.5 / 8)
    assert (s[-1].double() - w).abs().max() <= tol and (s1[0].double() - w).abs().max() <= tol


@pytest.mark.parametrize("n", [20, 70, 200])
def test_vanishing_reflectors(n):
    # a diagonal matrix, a tridiagonal one, the zero matrix, and a rank-one matrix: columns whose
    # norm below the diagonal (or whole) is zero, or rounding noise whose squares underflow
    d = torch.diag(torch.linspace(1.0, -2.0, n))
    t = d + torch.diag(torch.full((n - 1,), 0.25), 1) + torch.diag(torch.full((n - 1,), 0.25), -1)
    u = torch.ones(n, 1) / n ** 0.5
    _check(torch.stack([d, t, torch.zeros(n, n), u @ u.T, 1e-12 * (u @ u.T)]).cuda())


@pytest.mark.parametrize("n", [2, 3, 4, 15, 16, 17, 18, 31, 32, 33, 34, 35, 48, 49, 255, 256, 257, 258])
@pytest.mark.parametrize("gap", [1e-2, 1e-7])
def test_inverse_iteration_halves(n, gap):
    """Inverse iteration works from both ends of T towards the middle, 8 rows to a stage, 16 vectors to a
    warp: odd and even sizes around those, with all eigenvalues apart (float-float) and in pairs
    1e-7 apart (FP64)."""
    g = torch.Generator()
    g.manual_seed(n)
    q = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=torch.float64))[0]
    lam = torch.linspace(1.0, -1.0, n, dtype=torch.float64) if gap > 1e-3 else \
        torch.linspace(1.0, -1.0, (n + 1) // 2, dtype=torch.float64).repeat_interleave(2)[:n]
    if gap < 1e-3:
        lam = lam + gap * (torch.arange(n, dtype=torch.float64) % 2)
    h = (q * lam) @ q.T
    _check(torch.stack([h, -3.0 * h]).float().cuda())


@pytest.mark.parametrize("batch,n", [(1, 255), (10, 511), (20, 500), (37, 512), (75, 512), (150, 520)])
def test_multisection_lanes(batch, n):
    # 32, 16, 8, 4 and 2 lanes per eigenvalue, blocks with a remainder, eigenvalues apart and in pairs (refined)
    g = torch.Generator()
    g.manual_seed(n)
    q = torch.linalg.qr(torch.randn(n, n, generator=g, dtype=torch.float64))[0]
    lam = torch.linspace(1.0, -1.0, n, dtype=torch.float64)
    pairs = lam[::2].repeat_interleave(2)[:n] + 1e-7 * (torch.arange(n, dtype=torch.float64) % 2)
    h = torch.stack([(q * lam) @ q.T, (q * pairs) @ q.T]).float().cuda()
    h = h.repeat((batch + 1) // 2, 1, 1)[:batch].contiguous()
    _check(h)
    import paper_2609_32505_gb300 as P
    s = P.eigh(h)[0].double()
    for b in range(min(2, batch)):
        w = torch.linalg.eigvalsh(h[b].double()).flip(-1)
        assert (s[b::2] - w).abs().max() <= 2e-6 * max(1.0, n ** 0.5 / 8)
