"""Programmatic dependent launch: a kernel that lets its successor start early must wait for its own predecessor
on every path, also where it has nothing to do, or its completion no longer stands for that of the launches
before it (the counters a later pass resets, a graph's next node, a workspace that is handed on)."""
import ctypes
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32505_gb300", "csrc")


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


def test_every_path_waits_for_the_launch_before():
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = _code(path)
        for at in [m.start() for m in re.finditer(r"griddepcontrol\.launch_dependents", text)]:
            wait = text.find("griddepcontrol.wait", at)
            assert wait > 0, path
            between = text[at:wait]
            assert not re.search(r"\b(return|if|for|while)\b", between), (path, between)
            seen += 1
    assert seen > 0


def test_epilogues_do_not_read_through_the_read_only_path():
    # the in-place epilogues of the product kernel overwrite what they read; the non-coherent path is only for
    # memory that nothing writes while the kernel runs
    for name in ("gemm.cuh", "ops.cuh"):
        text = _code(os.path.join(CSRC, name))
        assert "global.nc" not in text and "__ldg" not in text, name


def test_shared_memory_limits_do_not_depend_on_the_call():
    # the limit is the function's, for every thread: a value that goes with the call's sizes could be lowered by another
    # thread between a call's setting and its launch
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = _code(path)
        for m in re.finditer(r"cudaFuncAttributeMaxDynamicSharedMemorySize,([^;]*?)\)\s*[;)]", text):
            names = set(re.findall(r"[A-Za-z_][A-Za-z_0-9.]*", m.group(1))) - {"int", "sizeof", "Sm"}
            assert all(re.fullmatch(r"k[A-Z]\w*", x) for x in names), (path, m.group(0))
            seen += 1
    assert seen >= 10


@pytest.mark.gpu
def test_captured_rerun_matches_stream():
    # a learned schedule whose bounds are far off for one matrix: its rerun resets the counters that the
    # first pass's last launches read.  Captured into a graph and replayed, the bits are those of the stream.
    import torch

    import paper_2609_32505_gb300 as P
    import workloads as W
    a = torch.stack([torch.from_numpy(W.constructed(70 + b, 300, 200, W.kappa_spectrum(200, 100.0))[0]).float()
                     for b in range(3)]).cuda()
    lb = torch.tensor([1e-3, 0.9, 1e-3], device="cuda")
    o = P.make_opts(schedule=P.SCHED_LEARNED, lower_bound=lb)
    w0, h0, info = P.polar(a, o, return_info=True)
    assert [i["status"] for i in info] == [0, 0, 0] and info[1]["sched_fallback"] == 1
    L = P.lib()
    w, h = torch.empty_like(w0), torch.empty_like(h0)
    ws = torch.empty(L.psvd_polar_workspace_bytes(3, 300, 200, ctypes.byref(o)), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert L.psvd_polar_fwd(P._ptr(a), P._ptr(w), P._ptr(h), 3, 300, 200, ctypes.byref(o), P._ptr(ws), ws.numel(),
                                None, P._stream()) == 0
    for _ in range(5):
        w.fill_(float("nan"))
        ws.fill_(255)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(w, w0) and torch.equal(h, h0)
