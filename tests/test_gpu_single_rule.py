"""Which launches at 16 lanes per cell solve every cell alone on a warp: the share
of the resident warps that the pairs may fill, on each side of its lines."""
import pytest

import synth
from tests.test_gpu_capture import _captured

pytestmark = pytest.mark.gpu


# rows, twelfths of the resident warps
@pytest.mark.parametrize("n,share", [(41, 4), (48, 4), (49, 9), (80, 9)])
def test_share_of_the_warps_that_pairs_may_fill(cuda, n, share):
    import torch
    from paper_2405_17363_gb300 import camp
    m = synth.make_mechanism(n, 2 * n, 800 + n)
    cb = synth.make_cells(m, 5000, 801 + n, gamma=(1e-4, 1e-1))
    A, b = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b))
    s = camp.Solver(m.row_ptr, m.col_idx)
    s.set_ordering(0)
    s.set_single_tail(0)
    want = [t.clone() for t in s.solve(A, b)]
    (pairs, grid, block, _), = _captured(lambda: s.solve(A, b))
    resident = grid[0] * block[0] // 32
    assert resident < 2500
    s.set_single_tail(-1)
    most = 2 * (share * resident // 12)
    for cells, alone in ((most - 1, True), (most, True), (most + 1, False)):
        (kernel, _, _, _), = _captured(lambda: s.solve(A[:cells], b[:cells]))
        assert (kernel != pairs) == alone
        for x, y in zip(s.solve(A[:cells], b[:cells]), want):
            assert torch.equal(x.view(torch.int32), y[:cells].view(torch.int32))
    s.close()
