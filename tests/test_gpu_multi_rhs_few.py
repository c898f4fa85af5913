"""Solves with a few right-hand sides on FP32 grids, whose level-0 sweeps run on copies of the rows in
shared memory: one part of the columns and several, full and ragged, odd numbers of them (padded rows
behind), block sizes beyond the shared memory that needs no opt-in, odd and even numbers of grid columns
(a last row without a neighbour, a last kept row without an eliminated one), and counts on either side
of where a thread per row and column takes over.  Every column's residual is formed with the operator."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402


@pytest.mark.parametrize("cells,px,ny,nrhs", [(1, 1, 34, 2), (3, 5, 48, 3), (3, 8, 224, 2), (2, 7, 256, 33),
                                              (4, 8, 64, 32), (5, 5, 100, 65), (10, 8, 160, 7),
                                              (62, 8, 48, 128), (62, 8, 48, 129)])
def test_every_column_is_solved(cells, px, ny, nrhs):
    d = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    with P.Grid(d, prec=P.FP32_REFINE) as g:
        g.set_design(W.widths(cells, ny, lo=0.02 * px, hi=0.045 * px))
        g.factor()
        torch.manual_seed(nrhs)
        b = torch.randn(g.N * nrhs, dtype=torch.complex128, device="cuda")
        x, info = g.solve(b, nrhs)
        assert not info.fallback and not info.simt_refactor
        B, X = b.view(g.N, nrhs), x.view(g.N, nrhs)
        for q in range(nrhs):
            r = B[:, q] - g.apply_operator(X[:, q].contiguous())
            assert float(r.norm() / B[:, q].norm()) <= 1.01e-10
        # one refinement step at most is left to the first solve's error
        g.set_refinement(1e-2, 0)
        _, first = g.solve(b, nrhs)
        assert first.rel_residual < 1e-3 and not first.fallback
