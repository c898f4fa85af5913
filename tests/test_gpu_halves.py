"""FP32 blocks of more than 160 rows, inverted by halves with one Newton step: sizes at both ends of
its range and beside them, halves of equal and of different sizes, grids of one batch and of a few
columns.  The first solve on the factorisation (no refinement step) has to be as accurate as FP32
rounding leaves it, and the refined value has to match the oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402
from oracle.reciprocal import Evaluation  # noqa: E402


@pytest.mark.parametrize("cells,px,ny", [(3, 8, 160), (3, 8, 162), (4, 5, 176), (3, 7, 190), (6, 8, 224),
                                         (2, 8, 248), (2, 8, 250)])
def test_first_solve_and_refined_value(cells, px, ny):
    d = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    wl = W.Workload("halves", d, W.Objective(W.OBJ_PLANEWAVE, monitor_row=24, theta_out=0.1),
                    W.Light(W.LIGHT_CONE, c=0.3), 16)
    ws = W.widths(cells, ny, lo=0.02 * px, hi=0.045 * px)
    F_ref, _ = Evaluation(wl, ws).reciprocal()
    with P.Grid(d, prec=P.FP32_REFINE) as g:
        g.set_design(ws)
        g.factor()
        # FP32 products and inverses of condition up to some 1e3, a few levels: below 1e-2 by far
        g.set_refinement(1e-2, 0)
        _, first = g.avg_intensity(wl.objective, wl.light)
        assert first.rel_residual < 1e-3 and not first.simt_refactor and not first.fallback
        g.set_refinement(1e-10, 30)
        F, info = g.avg_intensity(wl.objective, wl.light)
    assert not info.simt_refactor and not info.fallback
    assert abs(F - F_ref) <= 1e-8 * abs(F_ref), (F, F_ref)
