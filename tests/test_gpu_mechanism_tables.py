"""The mechanism tables of the fused assembly and the Newton corrector where they
can go wrong: more reactions than a cell's matrix block holds rates (several
chunks), first- and second-order reactions in any order (constant terms in the
middle of a chain), fewer chains than lanes, and every lane count, against the
oracle's plain-C assembly, solve and Newton loop with the bars of their tests."""
import numpy as np
import pytest

import oracle
import synth
from tests import parity
from tests.test_gpu_newton import NEWTON_TOL, _compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,lanes", [(3, 5, 1), (3, 40, 32), (5, 150, 2), (8, 200, 8), (8, 3, 16),
                                       (21, 60, 4), (40, 90, 8), (57, 400, 16), (80, 200, 16),
                                       (100, 230, 32)])
def test_tables_match_oracle(cuda, n, R, lanes):
    import torch
    from paper_2405_17363_gb300 import camp
    m = synth.make_mechanism(n, R, 300 + n)
    cb = synth.make_cells(m, 203, 400 + n, gamma=(1e-4, 1e-1))
    p = np.random.default_rng(n).permutation(R)
    args = (m.reactants[p, 0], m.reactants[p, 1], m.products[p], m.k[p])
    s = camp.Solver(m.row_ptr, m.col_idx)
    s.set_arrangement(camp.CAMP_ARR_WARP, lanes, 1, 0)
    s.set_mechanism(*args)
    conc, gam, b = (torch.as_tensor(v, device=cuda) for v in (cb.conc, cb.gamma, cb.b))
    x, it, res, st = s.assemble_solve(conc, gam, b, 1e-10, 500)
    out = s.newton_solve(conc, gam, conc, newton_tol=NEWTON_TOL)
    torch.cuda.synchronize()
    s.close()
    A = oracle.assemble(m.row_ptr, m.col_idx, *args, cb.conc, cb.gamma)
    orc = oracle.solve(m.row_ptr, m.col_idx, A, cb.b, 1e-10, 500, threads=8)
    gpu = dict(x=x.cpu().numpy(), iters=it.cpu().numpy(), resid=res.cpu().numpy(),
               status=st.cpu().numpy())
    parity.compare(m, A, cb.b, 1e-10, gpu, orc, f"tables n{n} R{R} lanes{lanes}")
    no = oracle.newton(m.row_ptr, m.col_idx, *args, cb.conc, cb.gamma, cb.conc.copy(),
                       newton_tol=NEWTON_TOL)
    _compare({k: v.cpu().numpy() for k, v in out.items()}, no, f"newton n{n} R{R} lanes{lanes}")
