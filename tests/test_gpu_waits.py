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


def _two_levels():
    """Two levels in L, one in U (few levels: streamed): 20,480 rows of their
    diagonal alone, then 30,752 rows with 116 entries among those, the widest
    that are streamed.  With 32 CTAs the second level's 961 slices are shares
    of 31, one slice to a tile: one CTA has none and waits for all the others."""
    n0, n1, w = 20480, 961 * 32, 116
    rng = np.random.default_rng(83)
    col = np.sort((rng.integers(0, n0, size=(n1, 1)) + 176 * np.arange(w)) % n0, axis=1)
    wide = np.concatenate([col, n0 + np.arange(n1)[:, None]], axis=1)
    val = np.concatenate([rng.uniform(-1.0, 1.0, size=(n1, w)) / w, np.full((n1, 1), 2.0)], axis=1)
    rp = np.concatenate([np.arange(n0), n0 + (w + 1) * np.arange(n1 + 1)]).astype(np.int64)
    return W.CSR(row_ptr=rp, col=np.concatenate([np.arange(n0), wide.ravel()]).astype(np.int32),
                 val=np.concatenate([np.full(n0, 2.0), val.ravel()]), n_rows=n0 + n1)


def _band(N, half, cplx=False):
    """A band whose rows all depend on the row before: one row to a level."""
    r, c = np.meshgrid(np.arange(N), np.arange(-half, half + 1), indexing="ij")
    keep = (r + c >= 0) & (r + c < N)
    v = np.where(c == 0, 3.0, -1.0 / (half * (1.0 + np.abs(c))) * (1.0 + 0.3 * np.sign(c)))
    if cplx:
        v = v * (1.0 + 0.25j)
    rp = np.concatenate([[0], np.cumsum(keep.sum(axis=1))]).astype(np.int64)
    return W.CSR(row_ptr=rp, col=(r + c)[keep].astype(np.int32), val=v[keep], n_rows=N)


def _solve_or_timeout(solve, limits):
    """solve(limit) -> results; how many limits ended in MLB_ERR_TIMEOUT.
    The other calls, the one with the longest limit among them, must be right."""
    ended = 0
    for limit in limits:
        try:
            results = solve(limit)
        except M.MlbError as e:
            assert e.code == M.MLB_ERR_TIMEOUT and limit != limits[-1], limit
            ended += 1
            continue
        assert all(r.status == 0 and r.flag == 0 and r.true_relres < 1e-9 for r in results), limit
    return ended


LIMITS = [1, 3_000, 30_000, 100_000, 300_000, 1_000_000, 2_000_000_000]


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("kind,precond,grid,must_end", [
    ("two levels", M.MLB_PRECOND_ILU0, 32, True),    # streamed levels
    ("band", M.MLB_PRECOND_ILU0, 7, True),           # values by slots
    ("complex band", M.MLB_PRECOND_ILU0, 7, False),  # a barrier per level
    ("complex band", M.MLB_PRECOND_ILU0_MC, 7, False),
    ("stencil", M.MLB_PRECOND_ILU0_MC, 23, False),
    ("stencil", M.MLB_PRECOND_NONE, 23, False),
    ("stencil", M.MLB_PRECOND_NONE, 1, False),
])
def test_waits_that_run_out_end_the_solve(kind, precond, grid, must_end, precision):
    """With limits from a nanosecond on, some wait of a working solve runs out
    first: at a level of M^{-1} (a CTA without rows there, a chain of rows), at
    a team sum, at a tile.  Wherever that is, the call returns
    MLB_ERR_TIMEOUT, or the solution, and the next call works."""
    A = {"two levels": _two_levels, "band": lambda: _band(6000, 40),
         "complex band": lambda: _band(1500, 12, cplx=True),
         "stencil": lambda: W.cd3d_lognormal(24, sigma=1.0)}[kind]()
    b = W.uniform_rhs(A.n_rows, seed=84).astype(A.val.dtype)

    def solve(limit):
        h = M.mlbicgstab_create(A, n=3, q_seed=0, precond=precond, precision=precision, grid=grid, timeout_ns=limit)
        try:
            return [M.mlbicgstab_solve(h, b, np.zeros_like(b), 1e-9, 4000)[0]]
        finally:
            h.destroy()

    ended = _solve_or_timeout(solve, LIMITS)
    if must_end:
        assert ended > 0


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("precond", [M.MLB_PRECOND_NONE, M.MLB_PRECOND_ILU0, M.MLB_PRECOND_ILU0_MC])
def test_waits_that_run_out_end_a_batch(precond, precision):
    """The same for a batch, where a CTA goes on to the next system after one
    that a wait ended."""
    systems = [W.cd3d_lognormal(m, sigma=1.0) for m in (24, 22, 6, 9, 12, 7, 10, 5, 11, 8)]
    bs = [W.uniform_rhs(A.n_rows, seed=85) for A in systems]

    def solve(limit):
        hs = [M.mlbicgstab_create(A, n=3, q_seed=0, precond=precond, precision=precision, timeout_ns=limit)
              for A in systems]
        try:
            return M.mlbicgstab_solve_batch(hs, bs, [np.zeros_like(b) for b in bs], [1e-9] * len(hs),
                                            [4000] * len(hs))
        finally:
            for h in hs:
                h.destroy()

    _solve_or_timeout(solve, LIMITS)


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("kind,N", [("real", 60000), ("complex", 30000)])
def test_long_triangular_solves_are_no_timeout(kind, N, precision):
    """A chain of N levels in each triangle, a microsecond or more each: one
    M^{-1} (tens of milliseconds) lasts many times the limit of 5 ms, which no
    single wait of a level comes near.  ILU(0) of a tridiagonal matrix is exact,
    so that few iterations solve it."""
    A = _band(N, 1, cplx=kind == "complex")
    xs = W.uniform_rhs(N, seed=86).astype(A.val.dtype)
    rows = np.repeat(np.arange(N), np.diff(A.row_ptr))
    b = np.zeros_like(xs)
    np.add.at(b, rows, A.val * xs[A.col])
    h = M.mlbicgstab_create(A, n=2, q_seed=0, precond=M.MLB_PRECOND_ILU0, precision=precision, timeout_ns=5_000_000)
    x = np.zeros_like(b)
    r, _ = M.mlbicgstab_solve(h, b, x, 1e-11, 50)
    assert r.flag == 0 and r.true_relres < 1e-11
    # at least two M^{-1}, each longer than twice the limit
    assert r.kernel_ms > 2 * 2 * 5.0
    # diagonally dominant, ||A^-1||_2 <= 1 / (|d| - off-diagonal sum)
    d = np.abs(A.val[rows == A.col]).min()
    off = np.zeros(N)
    np.add.at(off, rows[rows != A.col], np.abs(A.val[rows != A.col]))
    offc = np.zeros(N)
    np.add.at(offc, A.col[rows != A.col], np.abs(A.val[rows != A.col]))
    gap = d - 0.5 * (off.max() + offc.max())
    assert gap > 0
    assert np.linalg.norm(x - xs) <= 1.1e-11 * np.linalg.norm(b) / gap
    h.destroy()


def test_selftest_makes_every_wait_between_ctas_run_out():
    """The counter barrier, a team sum and a value slot, one after another:
    three limits pass before the answer."""
    import time
    M.mlbicgstab_selftest_barrier_timeout(4, 1_000_000)
    t = time.perf_counter()
    assert M.mlbicgstab_selftest_barrier_timeout(4, 60_000_000) == M.MLB_ERR_TIMEOUT
    assert time.perf_counter() - t >= 3 * 0.060
