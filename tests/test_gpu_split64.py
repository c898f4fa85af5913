"""The FP64 factorisation on the tensor cores (digit-split products, block inverses by Newton
iteration): solves without any refinement step, so that the factorisation's own error shows,
at block sizes below one tile, at its edges and beside them, odd, at the largest that the split
takes and one beyond (the general kernels); and blocks outside the FP32 range, whose Newton
iteration cannot start, so that the Gauss-Jordan kernel takes over."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402
from oracle.reciprocal import Evaluation  # noqa: E402

# A backward error of FP64 rounding: a few hundred roundings (levels x the terms of a sum) of
# 1.1e-16 each.  A single product that kept only the high digits would leave 1e-11 or more.
UNREFINED = 1e-12


def _workload(cells, ny, px=8, **kw):
    g = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6, **kw)
    return W.Workload("split", g, W.Objective(W.OBJ_PLANEWAVE, monitor_row=24, theta_out=0.1),
                      W.Light(W.LIGHT_CONE, c=0.3), 16)


def _unrefined(wl, ws, max_steps=0):
    with P.Grid(wl.grid, prec=P.FP64) as g:
        g.set_refinement(1e-13, max_steps)
        g.set_design(ws)
        g.factor()
        F, info = g.avg_intensity(wl.objective, wl.light)
        torch.manual_seed(1)
        b = torch.randn(g.N, dtype=torch.complex128, device="cuda")
        _, ib = g.solve(b)
    return F, info.rel_residual, ib.rel_residual


@pytest.mark.parametrize("cells,px,ny", [(3, 8, 34), (2, 5, 63), (3, 8, 64), (3, 5, 65), (4, 8, 128),
                                         (3, 7, 131), (12, 8, 160), (3, 8, 161), (2, 8, 224),
                                         (2, 7, 247), (2, 8, 248), (2, 8, 249)])
def test_unrefined_solve_has_fp64_backward_error(cells, px, ny):
    wl = _workload(cells, ny, px)
    ws = W.widths(cells, ny, lo=0.02 * px, hi=0.045 * px)
    F, r, rb = _unrefined(wl, ws)
    assert r < UNREFINED and rb < UNREFINED, (r, rb)
    F_ref, _ = Evaluation(wl, ws).reciprocal()
    assert abs(F - F_ref) <= 1e-9 * abs(F_ref), (F, F_ref)


def test_blocks_outside_the_fp32_range():
    wl = _workload(4, 64, eps_pillar=1e39)
    ws = W.widths(4, 5)
    F_ref, _ = Evaluation(wl, ws).reciprocal()
    F, _, _ = _unrefined(wl, ws, max_steps=2)
    assert abs(F - F_ref) <= 1e-9 * abs(F_ref), (F, F_ref)
