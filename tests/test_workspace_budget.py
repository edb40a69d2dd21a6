"""Scratch of inverse iteration: whole matrices at a time, as many as fit 3 GB, one at least."""
import pytest

BUDGET = 3.0e9


def _iv_bytes(n):
    # five arrays of doubles, 16 vectors of half the matrix (and a stage more) to a warp, and FP32 vectors
    rows = ((n - 1) // 2 + 9 + 1) // 2 * 2
    return 5 * 8 * 32 * ((n + 15) // 16) * rows + 4 * n * n


@pytest.mark.parametrize("n", [17, 33, 100, 600, 4096])
def test_inverse_iteration_scratch_is_bounded(n):
    import paper_2609_32505_gb300 as P
    L = P.lib()
    ws = lambda b: L.psvd_eigh_workspace_bytes(b, n)
    fit = int(BUDGET // _iv_bytes(n))                             # matrices that fit
    many = min(65535, 4 * fit)
    # what one more matrix takes besides (from batches past 640, where nothing else changes with the batch)
    other = (ws(4000) - ws(2000)) / 2000 - (_iv_bytes(n) if fit >= 4000 else 0)
    assert ws(many) - many * other <= BUDGET + 64e6
    assert fit >= (4 if n == 4096 else 1)
