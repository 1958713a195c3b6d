"""Calls made while their stream captures a graph: what they leave in the handle,
and which kernels a graph holds, must not depend on the calls made before."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def camp(cuda):
    from paper_2405_17363_gb300 import camp as c
    return c


# 100 species: 25 slots per lane as built, 22 aligned; 150: 37 and 36
@pytest.mark.parametrize("n,R", [(100, 250), (150, 400)])
@pytest.mark.parametrize("newton", [False, True])
def test_mechanism_tables_built_in_a_relaxed_capture(camp, cuda, n, R, newton):
    """The refinement prepares the lane count, a capture in relaxed mode (where
    allocation is allowed) makes the first fused call: its replays and the eager
    calls after it give bitwise the results of a handle that never captured."""
    import torch
    m = synth.make_mechanism(n, R, 500 + n)
    cb = synth.make_cells(m, 64, 501 + n, gamma=(1e-4, 1e-1))
    A, b, conc, gam = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b, cb.conc, cb.gamma))

    def handle():
        s = camp.Solver(m.row_ptr, m.col_idx)
        s.set_mechanism(m.reactants[:, 0], m.reactants[:, 1], m.products, m.k)
        return s

    def fused(s):
        if newton:
            return tuple(s.newton_solve(conc, gam, conc).values())
        return s.assemble_solve(conc, gam, b)

    ref = handle()
    want = [t.clone() for t in fused(ref)]
    s = handle()
    s.solve_mixed(A, b)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        captured = fused(s)
    g.replay()
    eager = fused(s)
    torch.cuda.synchronize()
    for x, y, z in zip(want, captured, eager):
        assert torch.equal(x.view(torch.int32), y.view(torch.int32))
        assert torch.equal(x.view(torch.int32), z.view(torch.int32))
    del g, captured
    s.close()
    ref.close()


def _kernel_nodes(graph):
    """(name, grid, block, dynamic shared memory) of the graph's kernel nodes."""
    import ctypes
    cu = ctypes.CDLL("libcuda.so.1")
    u, p = ctypes.c_uint, ctypes.c_void_p

    class Params(ctypes.Structure):
        _fields_ = [("func", p), ("grid", u * 3), ("block", u * 3), ("smem", u), ("params", p),
                    ("extra", p), ("kern", p), ("ctx", p)]

    raw, count = p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert cu.cuGraphGetNodes(raw, None, ctypes.byref(count)) == 0
    nodes = (p * count.value)()
    assert cu.cuGraphGetNodes(raw, nodes, ctypes.byref(count)) == 0
    got = []
    for q in nodes:
        kind, k, name = ctypes.c_int(), Params(), ctypes.c_char_p()
        assert cu.cuGraphNodeGetType(p(q), ctypes.byref(kind)) == 0
        if kind.value != 0:
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(p(q), ctypes.byref(k)) == 0
        if k.func:
            assert cu.cuFuncGetName(ctypes.byref(name), p(k.func)) == 0
        else:
            assert cu.cuKernelGetName(ctypes.byref(name), p(k.kern)) == 0
        got.append((name.value.decode(), tuple(k.grid), tuple(k.block), k.smem))
    return got


def _captured(call):
    import torch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    return _kernel_nodes(g)


def test_captured_refinement_runs_the_refinement_layout(camp, cuda):
    """solve_mixed captured after a solve launches what it launches eagerly (the
    schedule as built: its shared memory holds one slot per lane more)."""
    import torch
    m = synth.make_mechanism(100, 250, 600)
    cb = synth.make_cells(m, 64, 601, gamma=(1e-4, 1e-1))
    A, b = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b))
    nodes = []
    for first in ("solve", "solve_mixed"):
        s = camp.Solver(m.row_ptr, m.col_idx)
        getattr(s, first)(A, b)
        nodes.append(_captured(lambda: s.solve_mixed(A, b)))
        s.close()
    assert nodes[0] and nodes[0] == nodes[1]


@pytest.mark.parametrize("transpose", [False, True])
def test_captured_small_batch_runs_single_cells(camp, cuda, transpose):
    """A small batch at 16 lanes per cell, captured after one large solve, launches
    what it launches eagerly: every cell alone on a warp."""
    import torch
    m = synth.make_mechanism(80, 200, 602)
    cb = synth.make_cells(m, 5000, 603, gamma=(1e-4, 1e-1))
    A, b = (torch.as_tensor(v, device=cuda) for v in (cb.A_vals, cb.b))
    nodes = []
    for first in (5000, 64):
        s = camp.Solver(m.row_ptr, m.col_idx)
        s.solve(A[:first], b[:first], transpose=transpose)
        nodes.append(_captured(lambda: s.solve(A[:64], b[:64], transpose=transpose)))
        s.set_single_tail(0)
        pairs = _captured(lambda: s.solve(A[:64], b[:64], transpose=transpose))
        s.close()
    assert nodes[0] and nodes[0] == nodes[1] and nodes[0] != pairs
