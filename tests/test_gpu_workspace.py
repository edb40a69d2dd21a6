"""What a call returns does not depend on what its workspace held before: the same call through the C ABI
with a workspace of zero bytes and of 0xFF bytes (NaN in every float format) gives the same bits.  Sizes
with ragged tiles, more than one QR block and panel, and phases of the on-chip tridiagonalization."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def _both(nbytes, call):
    out = []
    for fill in (0, 255):
        ws = torch.full((max(int(nbytes), 256),), fill, dtype=torch.uint8, device="cuda")
        out.append([x.clone() for x in call(ws)])
    for x, y in zip(*out):
        assert torch.isfinite(x.float()).all()
        assert torch.equal(x, y)


def _mat(seed, *shape):
    g = torch.Generator()
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g).cuda()


@pytest.mark.parametrize("batch,m,n", [(1, 129, 129), (2, 300, 200), (2, 7000, 150), (3, 90, 40)])
def test_qr(batch, m, n):
    import paper_2609_32505_gb300 as P
    L = P.lib()
    a = _mat(m + n, batch, m, n)
    q, r = torch.empty_like(a), torch.empty(batch, n, n, device="cuda")

    def call(ws):
        assert L.psvd_qr(P._ptr(a), P._ptr(q), P._ptr(r), batch, m, n, P._ptr(ws), ws.numel(), P._stream()) == 0
        return q, r
    _both(L.psvd_qr_workspace_bytes(batch, m, n), call)


@pytest.mark.parametrize("batch,n", [(2, 3), (3, 130), (1, 700), (1, 1027), (1, 2100)])
def test_eigh(batch, n):
    import paper_2609_32505_gb300 as P
    L = P.lib()
    a = _mat(n, batch, n, n)
    h = (a + a.transpose(1, 2)).contiguous()
    s, vt = torch.empty(batch, n, device="cuda"), torch.empty_like(h)

    def call(ws):
        assert L.psvd_eigh(P._ptr(h), P._ptr(s), P._ptr(vt), batch, n, P._ptr(ws), ws.numel(), P._stream()) == 0
        return s, vt
    _both(L.psvd_eigh_workspace_bytes(batch, n), call)


@pytest.mark.parametrize("precision,preqr", [(0, 0), (1, 0), (2, 0), (1, 1)])
@pytest.mark.parametrize("batch,m,n", [(2, 300, 200), (1, 520, 257)])
def test_svd_fwd_bwd(batch, m, n, precision, preqr):
    import paper_2609_32505_gb300 as P
    L = P.lib()
    a = _mat(m, batch, m, n)
    u, s, vt = torch.empty_like(a), torch.empty(batch, n, device="cuda"), torch.empty(batch, n, n, device="cuda")
    o = P.make_opts(precision=precision, preqr=preqr)

    def fwd(ws):
        assert L.psvd_svd_fwd(P._ptr(a), P._ptr(u), P._ptr(s), P._ptr(vt), batch, m, n, ctypes.byref(o), P._ptr(ws),
                              ws.numel(), None, P._stream()) == 0
        return u, s, vt
    _both(L.psvd_svd_workspace_bytes(batch, m, n, ctypes.byref(o)), fwd)
    da, du, ds, dvt = torch.empty_like(a), _mat(1, batch, m, n), _mat(2, batch, n), _mat(3, batch, n, n)

    def bwd(ws):
        assert L.psvd_svd_bwd(P._ptr(a), P._ptr(u), P._ptr(s), P._ptr(vt), P._ptr(du), P._ptr(ds), P._ptr(dvt),
                              P._ptr(da), batch, m, n, 1e-8, 0, P._ptr(ws), ws.numel(), P._stream()) == 0
        return (da,)
    _both(L.psvd_svd_bwd_workspace_bytes(batch, m, n), bwd)
