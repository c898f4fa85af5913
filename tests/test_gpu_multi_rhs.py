"""Solves with several right-hand sides (all levels in one array, products over two segments):
numbers of right-hand sides at the edges of the column tiles, odd ones (padded columns in FP32),
even and odd numbers of rows at every level, block sizes beyond one row or column tile and beyond
what the FP64 split takes.  Every column's residual is formed again with the operator; FP64 solves
run without a refinement step, so that the substitution's own error shows (a few hundred
roundings of 1.1e-16)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2207_10701_gb300 as P  # noqa: E402
import workloads as W  # noqa: E402


def _residuals(g, b, x, nrhs):
    B, X = b.view(g.N, nrhs), x.view(g.N, nrhs)
    out = []
    for q in range(nrhs):
        r = B[:, q] - g.apply_operator(X[:, q].contiguous())
        out.append(float(r.norm() / B[:, q].norm()))
    return max(out)


def _grid(cells, px, ny, prec):
    d = W.GridDesc(n_cells=cells, ny=ny, cell_px=px, npml=8, rows_sub=6, rows_pillar=6)
    g = P.Grid(d, prec=prec)
    g.set_design(W.widths(cells, ny, lo=0.02 * px, hi=0.045 * px))
    g.factor()
    return g


CASES = [(3, 8, 48, 2), (3, 5, 64, 3), (2, 5, 66, 7), (4, 8, 80, 33), (3, 7, 130, 64), (5, 8, 160, 81),
         (3, 8, 162, 160), (2, 8, 224, 161), (3, 8, 96, 255), (2, 5, 48, 256)]


@pytest.mark.parametrize("cells,px,ny,nrhs", CASES)
@pytest.mark.parametrize("prec", [P.FP64, P.FP32_REFINE])
def test_every_column_is_solved(cells, px, ny, nrhs, prec):
    g = _grid(cells, px, ny, prec)
    if prec == P.FP64:
        g.set_refinement(1e-13, 0)
    torch.manual_seed(nrhs)
    b = torch.randn(g.N * nrhs, dtype=torch.complex128, device="cuda")
    for _ in range(2):                       # the second call on the workspace of the first
        x, info = g.solve(b, nrhs)
        tol = 1e-12 if prec == P.FP64 else 1.01e-10
        assert _residuals(g, b, x, nrhs) <= tol
        assert info.rel_residual <= tol and not info.fallback and not info.simt_refactor
    x1, _ = g.solve(b.view(g.N, nrhs)[:, 0].contiguous())     # one right-hand side afterwards
    assert _residuals(g, b.view(g.N, nrhs)[:, 0].contiguous(), x1, 1) <= tol
    g.close()


@pytest.mark.parametrize("ny,nrhs", [(249, 3), (251, 66)])
def test_fp64_blocks_beyond_the_split(ny, nrhs):
    g = _grid(2, 8, ny, P.FP64)
    g.set_refinement(1e-13, 0)
    torch.manual_seed(nrhs)
    b = torch.randn(g.N * nrhs, dtype=torch.complex128, device="cuda")
    x, _ = g.solve(b, nrhs)
    assert _residuals(g, b, x, nrhs) <= 1e-12
    g.close()
