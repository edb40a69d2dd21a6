"""Calls of different sizes from several host threads, each with its own stream: every one succeeds, with the bits it
has alone (a kernel's shared-memory limit belongs to the function, not to the call)."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_eigh_of_different_sizes_from_several_threads():
    import paper_2609_32505_gb300 as P
    sizes = [140, 250, 100, 181]
    hs, alone = [], []
    for n in sizes:
        g = torch.Generator()
        g.manual_seed(n)
        a = torch.randn(n, n, generator=g).cuda()
        hs.append(a + a.T)
        alone.append([x.clone() for x in P.eigh(hs[-1])])
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(200):
                    s, vt = P.eigh(hs[i])
                torch.cuda.current_stream().synchronize()
                assert torch.equal(s, alone[i][0]) and torch.equal(vt, alone[i][1])
        except Exception as e:                    # noqa: BLE001 (reported below, in the main thread)
            errors.append((sizes[i], repr(e)))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
