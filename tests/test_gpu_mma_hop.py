"""The tensor-core stencil of the FP16 solves at the edges of its tiles.

Blocks of the stencil work on 2 x 2 rows (y, z) of up to 4 half-sites in x for
groups of 8 sources, so the sizes below have rows of 1, 2, 3, 4, 5, 7 and 9
half-sites, the smallest extents (where a neighbour on both sides is the same
site), periodic and antiperiodic time, and 1 to 64 sources with a part-filled
last group.

Truncated solves (n CG iterations from zero, a fixed count) against the
oracle's in FP64.  Bound: every iteration stores six fields with unit roundoff
u = 2^-11 (p, t, w, t, r, x) and applies four hops whose links are rounded to u,
all of norm about one here (8 kappa ~ 1), so the solution's relative error is
at most about 10 n u; 16 n u is required normwise, and 64 n u of the largest
component at every site (a wrong neighbour is off by about 2 kappa).

(Tiles of 4 half-sites are those of the CG update; the hops of rows of 5, 6 and 9
to 12 half-sites run in tiles of up to 6.  Each block has one tile here;
test_gpu_mma_tiles.py has several.)
"""
import numpy as np
import pytest

from oracle import solver
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

KAPPA, MU, U16, N = 0.124, 0.01, 2.0 ** -11, 2


@pytest.mark.parametrize("dims,nrhs,apbc", [
    ((2, 2, 2, 2), 1, True), ((2, 4, 2, 4), 9, True), ((4, 2, 4, 2), 8, False), ((6, 4, 4, 4), 7, True),
    ((8, 4, 2, 4), 2, False), ((10, 4, 4, 2), 3, True), ((14, 2, 4, 4), 2, True), ((18, 4, 2, 2), 2, True)])
def test_truncated_solves_match_oracle(ctx, dims, nrhs, apbc):
    U = S.gauge_field(dims, 0.3, 5)
    ctx.load_gauge(U, dims, KAPPA, MU, antiperiodic_t=apbc)
    b = S.random_spinor(dims, 6, batch=(nrhs,))
    s, iters, _, _ = ctx.solve(b, tsm.stop(0.0, N, tsm.TSM_F16))
    assert np.all(iters == N)
    for r in range(nrhs):
        want = solver.solve_full(U, b[r], dims, KAPPA, MU, 0.0, N, apbc)[0]
        assert np.linalg.norm(s[r] - want) <= 16 * N * U16 * np.linalg.norm(want), r
        assert np.abs(s[r] - want).max() <= 64 * N * U16 * np.abs(want).max(), r


@pytest.mark.parametrize("nrhs", [33, 64])
def test_wide_batches_equal_single_solves(ctx, nrhs):
    """Part-filled and full groups, more groups than one: the same bits as alone."""
    dims = (6, 4, 4, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, KAPPA, MU)
    b = S.random_spinor(dims, 8, batch=(nrhs,))
    b[nrhs // 2] *= 1e-2
    stop = tsm.stop(5e-3, 60, tsm.TSM_F16)
    s, iters, _, _ = ctx.solve(b, stop)
    for r in (0, 8, nrhs // 2, nrhs - 1):
        one, it, _, _ = ctx.solve(b[r], stop)
        assert it[0] == iters[r] and np.array_equal(one, s[r]), r


@pytest.mark.parametrize("dims,nrhs,apbc", [
    ((12, 2, 4, 4), 9, True), ((12, 4, 2, 2), 17, False), ((22, 2, 2, 4), 2, True), ((24, 4, 4, 2), 5, True)])
def test_six_wide_tiles_match_oracle(ctx, dims, nrhs, apbc):
    """Rows of 6, 11 and 12 half-sites: the hops' tiles are 6 wide (6, 6 + 5 and
    6 + 6), the update's 3 and 4.  Bounds as above."""
    test_truncated_solves_match_oracle(ctx, dims, nrhs, apbc)
