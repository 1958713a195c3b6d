"""The first calls of a handle: the tables they upload are on the device before
any stream's kernel reads them, whichever stream that is."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def camp(cuda):
    from paper_2405_17363_gb300 import camp as c
    return c


# few and many entries: tables of a few KB and of several hundred
@pytest.mark.parametrize("n,R,cells", [(30, 60, 64), (80, 200, 300), (80, 200, 4000), (150, 400, 700),
                                       (100, 5000, 64)])
def test_first_call_on_a_side_stream(camp, cuda, n, R, cells):
    """Fresh handles whose first call runs on a stream that is not ordered behind
    the legacy stream give bitwise the results of a handle on the legacy stream."""
    import torch
    m = synth.make_mechanism(n, R, 500 + n)
    cb = synth.make_cells(m, cells, 501 + n, gamma=(1e-4, 1e-1))
    A, b, conc, gam = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b, cb.conc, cb.gamma))

    def calls(s):
        s.set_mechanism(m.reactants[:, 0], m.reactants[:, 1], m.products, m.k)
        return [lambda: s.solve(A, b), lambda: s.solve(A, b, transpose=True),
                lambda: s.solve_mixed(A, b), lambda: s.assemble_solve(conc, gam, b),
                lambda: tuple(s.newton_solve(conc, gam, conc).values())]

    side = torch.cuda.Stream()
    for q in range(5):
        ref = camp.Solver(m.row_ptr, m.col_idx)
        want = [t.clone() for t in calls(ref)[q]()]
        torch.cuda.synchronize()
        for _ in range(4):
            s = camp.Solver(m.row_ptr, m.col_idx)
            with torch.cuda.stream(side):
                got = calls(s)[q]()
            side.synchronize()
            for x, y in zip(want, got):
                assert torch.equal(x.view(torch.int32), y.view(torch.int32))  # the bits
            s.close()
        ref.close()
