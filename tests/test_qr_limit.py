"""The row limit of psvd_qr is the one its header states."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_header_and_code_agree():
    txt = open(os.path.join(ROOT, "include", "psvd.h")).read()
    stated = set(re.findall(r"m (?:<=|>) (\d{5})", txt))
    code = open(os.path.join(ROOT, "paper_2609_32505_gb300", "csrc", "qr.cuh")).read()
    assert stated == set(re.findall(r"kQrMaxRows = (\d+)", code))


def test_refusal_at_the_limit():
    # one row above the limit is refused before anything is launched; preqr falls back to the matrix itself there
    import paper_2609_32505_gb300 as P
    L = P.lib()
    fake = ctypes.c_void_p(1 << 20)
    assert L.psvd_qr(fake, fake, None, 1, 23025, 8, fake, 1 << 40, None) == -1
    o, plain = P.make_opts(preqr=1), P.make_opts()
    ws = lambda m, opts: L.psvd_polar_workspace_bytes(1, m, 8, ctypes.byref(opts))
    assert ws(23025, o) == ws(23025, plain) and ws(23024, o) != ws(23024, plain)


@pytest.mark.gpu
def test_preqr_on_either_side():
    import torch

    import paper_2609_32505_gb300 as P
    g = torch.Generator()
    g.manual_seed(3)
    for m in (23024, 23025):
        a = torch.randn(m, 20, generator=g).cuda()
        w, h, info = P.polar(a, P.make_opts(preqr=1), return_info=True)
        assert info[0]["status"] == 0
        assert (w.double() @ h.double() - a.double()).norm() <= 1e-5 * a.double().norm()
