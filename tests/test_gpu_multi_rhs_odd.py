"""FP64 solves with several right-hand sides at odd numbers of rows (within the digit split and above it),
unrefined, every column's residual formed again with the operator: a few hundred roundings of 1.1e-16."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402


@pytest.mark.parametrize("cells,px,ny,nrhs", [(3, 5, 33, 2), (2, 5, 63, 33), (3, 8, 65, 7), (3, 7, 131, 96),
                                              (2, 8, 161, 3), (2, 5, 247, 17), (2, 5, 249, 5)])
def test_every_column_is_solved(cells, px, ny, nrhs):
    d = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    with P.Grid(d, prec=P.FP64) as g:
        g.set_refinement(1e-13, 0)
        g.set_design(W.widths(cells, ny, lo=0.02 * px, hi=0.045 * px))
        g.factor()
        torch.manual_seed(nrhs)
        b = torch.randn(g.N * nrhs, dtype=torch.complex128, device="cuda")
        x, _ = g.solve(b, nrhs)
        B, X = b.view(g.N, nrhs), x.view(g.N, nrhs)
        for q in range(nrhs):
            r = B[:, q] - g.apply_operator(X[:, q].contiguous())
            assert float(r.norm() / B[:, q].norm()) <= 1e-12
