"""The virtual-focus row on narrow source planes: one column, one anchor's columns and beside them, as
many anchors as warps and one more, with the numbers of node chunks that low and high grids take
(a last chunk of fewer nodes among them)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402
from oracle.reciprocal import Evaluation  # noqa: E402


@pytest.mark.parametrize("cells,px,ny", [(1, 1, 34), (3, 5, 34), (9, 7, 40), (8, 8, 100), (13, 5, 127),
                                         (64, 8, 34), (27, 19, 64), (257, 8, 34), (3, 8, 160)])
def test_row_of_a_narrow_plane(cells, px, ny):
    g = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    obj = W.Objective(W.OBJ_VIRTUAL_FOCUS, monitor_row=23, x_f=0.4 * cells * px / g.ppl, d_rows=90)
    wl = W.Workload("vf", g, obj, W.Light(W.LIGHT_CONE, c=0.3), 16)
    ws = W.widths(cells, 3, lo=0.01 * px, hi=0.045 * px)
    F_ref, v_ref = Evaluation(wl, ws).reciprocal()
    with P.Grid(g, prec=P.FP64) as grid:
        grid.set_design(ws)
        grid.factor()
        F, _ = grid.avg_intensity(obj, wl.light)
        v, _ = grid.solve_reciprocal(obj)
    assert abs(F - F_ref) <= 1e-9 * abs(F_ref), (F, F_ref)
    err = abs(v.cpu().numpy() - v_ref).max() / abs(v_ref).max()
    assert err <= 1e-9, err
