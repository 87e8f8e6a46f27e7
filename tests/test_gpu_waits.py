"""Waits of the solve kernels: between consumers and producer where a pass has
no tiles, waits that run out, and long ones that must not."""
import numpy as np
import pytest

from paper_1106_3678_gb300 import mlbicgstab as M
from paper_1106_3678_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PRECISIONS = [M.MLB_PREC_FP64, M.MLB_PREC_FP32_REFINED]


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("kind,grid", [("few rows", 152), ("few rows", 17), ("wide rows", 7), ("wide rows", 152)])
def test_passes_without_tiles(kind, grid, precision):
    """A CTA without rows, or a product whose rows are too wide for a tile,
    gives the producer nothing to copy: only the counted ends of the passes
    keep the two sides together.  b = A x* is solved for x* as on one CTA."""
    A = W.cd2d(8) if kind == "few rows" else W.random_dense_system(200, seed=81)[0]
    N = A.n_rows
    D = np.zeros((N, N))
    D[np.repeat(np.arange(N), np.diff(A.row_ptr)), A.col] = A.val
    xs = W.uniform_rhs(N, seed=82)
    b = D @ xs
    # ||x - x*|| <= ||A^-1|| (||r|| + the rounding of b), ||r|| < tol ||b||
    tol = 1e-11
    bound = (tol + N * 2.3e-16) * np.linalg.norm(np.linalg.inv(D), 2) * np.linalg.norm(np.abs(D) @ np.abs(xs))
    for n in (1, 3):
        h = M.mlbicgstab_create(A, n=n, q_seed=0, precision=precision, grid=grid)
        for _ in range(3):
            x = np.zeros(N)
            r, _ = M.mlbicgstab_solve(h, b, x, tol, 2000)
            assert r.flag == 0 and r.true_relres < tol
            assert np.linalg.norm(x - xs) <= bound
        h.destroy()
