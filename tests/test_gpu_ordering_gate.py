"""Which launches order their cells: those whose groups do not all start at once,
or number more than one per SM sub-partition."""
import pytest

import synth
from tests.test_gpu_capture import _captured

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def camp(cuda):
    from paper_2405_17363_gb300 import camp as c
    return c


def _same(got, want):
    import torch
    return all(torch.equal(x.view(torch.int32), y.view(torch.int32)) for x, y in zip(got, want))


def test_cells_too_large_for_four_warps_are_ordered(camp, cuda):
    """7,100 entries leave room for two or three warps per SM: one cell more than
    start at once is ordered (mode 2 shows it as launches of its own), as many as
    start at once are not, and the results are bitwise those of index order."""
    import torch
    m = synth.make_mechanism(100, 5000, 700)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    cells = 4 * sms
    cb = synth.make_cells(m, cells, 701, gamma=(1e-4, 1.0))
    A, b, conc, gam = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b, cb.conc, cb.gamma))
    s = camp.Solver(m.row_ptr, m.col_idx)
    s.set_mechanism(m.reactants[:, 0], m.reactants[:, 1], m.products, m.k)
    s.set_ordering(0)
    want = [t.clone() for t in s.solve(A, b)]
    fused = [t.clone() for t in s.assemble_solve(conc, gam, b)]
    (_, grid, block, _), = _captured(lambda: s.solve(A, b))
    resident = grid[0] * block[0] // 32   # warps: the launch is as large as fits
    assert resident < cells
    s.set_ordering(2)
    assert _same(s.solve(A, b), want)
    for c, ordered in ((resident, False), (resident + 1, True), (cells, True)):
        nodes = _captured(lambda: s.solve(A[:c], b[:c]))
        assert any("classify" in k[0] for k in nodes) == ordered
    s.set_ordering(1)
    for _ in range(2):
        assert _same(s.solve(A, b), want) and _same(s.assemble_solve(conc, gam, b), fused)
    assert not s.get_fault()
    other = camp.Solver(m.row_ptr, m.col_idx)
    batch = camp.Batch([s, other])
    h = cells // 2
    got = batch.solve([A[:h], A[h:]], [b[:h], b[h:]])
    torch.cuda.synchronize()
    assert _same(got[0], [t[:h] for t in want]) and _same(got[1], [t[h:] for t in want])
    batch.close()
    other.close()
    s.close()


# (species, reactions, call, cells per warp): all rows sampled (up to 8 species),
# a sample of them, the refinement (several cells per warp), by gamma; single
# cells (16 lanes, small batch) are a warp each
@pytest.mark.parametrize("n,R,call,k", [(6, 12, "solve", 16), (30, 60, "solve", 4), (80, 200, "solve", 1),
                                        (24, 60, "solve_mixed", 4), (80, 200, "assemble_solve", 2)])
def test_small_ordered_launches_between_large_ones(camp, cuda, n, R, call, k):
    """One group more than starts at once is ordered and one group fewer is not;
    in a sequence of such launches and larger ones every mode gives bitwise the
    results of index order (nothing left over from a launch misplaces a cell)."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edge = 4 * sms * k
    sizes = (edge + 1, 5 * edge + 7, edge, edge + 1, 2 * edge + 3, edge + k)
    m = synth.make_mechanism(n, R, 710 + n)
    cb = synth.make_cells(m, max(sizes), 711 + n, gamma=(1e-4, 1e-1))
    A, b, conc, gam = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b, cb.conc, cb.gamma))
    s = camp.Solver(m.row_ptr, m.col_idx)
    s.set_mechanism(m.reactants[:, 0], m.reactants[:, 1], m.products, m.k)

    def run(c):
        if call == "assemble_solve":
            return s.assemble_solve(conc[:c], gam[:c], b[:c])
        return getattr(s, call)(A[:c], b[:c])

    s.set_ordering(0)
    want = [t.clone() for t in run(max(sizes))]
    for mode in (1, 2, 1):
        s.set_ordering(mode)
        for c in sizes:
            assert _same(run(c), [t[:c] for t in want]), (mode, c)
    assert not s.get_fault()
    if call != "assemble_solve":   # mode 2 of the others shows as launches of its own
        s.set_ordering(2)
        assert len(_captured(lambda: run(edge))) == 1
        assert any("classify" in q[0] for q in _captured(lambda: run(edge + 1)))
    s.close()
