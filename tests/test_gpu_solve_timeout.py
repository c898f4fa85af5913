"""An expired tensor-core wait in a solve with several right-hand sides is reported as such by the
factorisation that solved: the FP64 one of an FP64 grid, and the FP64 fallback of an FP32 grid (whose
own FP32 factorisation did not take part).  The wait runs out because its bound is lowered to a few
hundred cycles; the kernel returns and the grid works again with the default bound."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402

RCI_ETIMEOUT = 8


@pytest.mark.parametrize("prec", [P.FP64, P.FP32_REFINE])
def test_expired_wait_in_a_solve(prec):
    wl = W.small(kind=W.OBJ_VIRTUAL_FOCUS)
    with P.Grid(wl.grid, prec=prec) as g:
        if prec == P.FP32_REFINE:
            g.set_refinement(1e-10, 0)   # no refinement step: the FP32 solve does not do
        g.set_design(W.widths(wl.grid.n_cells, 13))
        g.factor()
        b = torch.randn(g.N * 3, dtype=torch.complex128, device="cuda")
        _, info = g.solve(b, 3)
        assert bool(info.fallback) == (prec == P.FP32_REFINE)
        P.set_wait_limit(300)
        try:
            with pytest.raises(P.RciError) as ei:
                g.solve(b, 3)
            assert ei.value.status == RCI_ETIMEOUT
        finally:
            P.set_wait_limit(0)
        g.factor()
        x, info = g.solve(b, 3)
        assert info.rel_residual < 1e-9


def test_expired_wait_in_an_fp64_factorisation():
    wl = W.small()
    with P.Grid(wl.grid, prec=P.FP64) as g:
        g.set_design(W.widths(wl.grid.n_cells, 13))
        P.set_wait_limit(300)
        try:
            with pytest.raises(P.RciError) as ei:
                g.factor()
            assert ei.value.status == RCI_ETIMEOUT
        finally:
            P.set_wait_limit(0)
        g.factor()
        _, info = g.avg_intensity(wl.objective, wl.light)
        assert info.rel_residual < 1e-9
