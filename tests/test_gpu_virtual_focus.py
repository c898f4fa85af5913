"""The virtual-focus objective row (anchored cosine sums) against the oracle's direct sums: source
planes of one anchor and less, exactly one, a ragged last one, more anchors than one block takes,
the fewer node chunks of low grids, and a focus beside the source plane.  The adjoint-free field
carries every entry of the row, so the averaged intensity is compared at the FP64 tolerance of
the parity tests."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402
from oracle.reciprocal import Evaluation  # noqa: E402


@pytest.mark.parametrize("cells,px,ny,at", [(1, 8, 48, 0.5), (8, 8, 48, 0.3), (9, 7, 72, 0.5),
                                            (13, 5, 48, -0.4), (258, 8, 48, 0.9)])
def test_virtual_focus_row(cells, px, ny, at):
    g = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    obj = W.Objective(W.OBJ_VIRTUAL_FOCUS, monitor_row=24, x_f=at * cells * px / g.ppl, d_rows=150)
    wl = W.Workload("vf", g, obj, W.Light(W.LIGHT_CONE, c=0.3), 16)
    ws = W.widths(cells, 3, lo=0.01 * px, hi=0.045 * px)
    F_ref, v_ref = Evaluation(wl, ws).reciprocal()
    with P.Grid(g, prec=P.FP64) as grid:
        grid.set_design(ws)
        grid.factor()
        for _ in range(2):      # the second call takes the stored quadrature rule
            F, _ = grid.avg_intensity(obj, wl.light)
            assert abs(F - F_ref) <= 1e-9 * abs(F_ref), (F, F_ref)
        v, _ = grid.solve_reciprocal(obj)
    err = abs(v.cpu().numpy() - v_ref).max() / abs(v_ref).max()
    assert err <= 1e-9, err
