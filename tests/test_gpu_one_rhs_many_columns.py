"""FP64 solves with one right-hand side on either side of the number of grid columns from which level 0
takes a thread instead of a warp per row: no refinement step, so that the substitution's own error shows
(a few hundred roundings of 1.1e-16)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402


@pytest.mark.parametrize("cells,px", [(302, 8), (1209, 2), (303, 8), (347, 7)])   # 1216, 1217, 1220, 1222 rows
def test_solve(cells, px):
    d = W.GridDesc(n_cells=cells, ny=34, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    with P.Grid(d, prec=P.FP64) as g:
        g.set_refinement(1e-13, 0)
        g.set_design(W.widths(cells, 5, lo=0.02 * px, hi=0.045 * px))
        g.factor()
        torch.manual_seed(cells)
        b = torch.randn(g.N, dtype=torch.complex128, device="cuda")
        x, _ = g.solve(b)
        r = b - g.apply_operator(x)
        assert float(r.norm() / b.norm()) <= 1e-12
