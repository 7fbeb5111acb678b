"""The tensor-core stencil's persistent blocks against the oracle: several tiles
per block (one block per SM), with the link words fetched one tile ahead, the
ring running on across tiles and groups, and the norms flushed every 8 tiles.

Truncated solves (n CG iterations from zero); bounds of test_gpu_mma_hop.py: 16 n u
normwise, 64 n u of the largest component (u = 2^-11).
"""
import numpy as np
import pytest

from oracle import philox, solver
from oracle.gamma import gamma_list
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

KAPPA, MU, U16 = 0.124, 0.01, 2.0 ** -11


@pytest.mark.parametrize("dims,nrhs,apbc", [
    ((8, 8, 8, 32), 9, True), ((4, 16, 16, 16), 9, False), ((2, 16, 16, 32), 3, True),
    ((12, 8, 8, 20), 9, True), ((10, 8, 10, 20), 17, False), ((18, 6, 6, 24), 9, True)])
def test_several_tiles_per_block(ctx, dims, nrhs, apbc):
    """Tiles of 4, 2 and 1 half-sites (512, 1024 and 2048 on 152 blocks) and hops in
    tiles of 6, 5 and 5 + 4 (320 to 432), a part-filled last group."""
    n = 2
    U = S.gauge_field(dims, 0.3, 5)
    ctx.load_gauge(U, dims, KAPPA, MU, antiperiodic_t=apbc)
    b = S.random_spinor(dims, 6, batch=(nrhs,))
    s, iters, _, _ = ctx.solve(b, tsm.stop(0.0, n, tsm.TSM_F16))
    assert np.all(iters == n)
    for r in (0, nrhs - 1):
        want = solver.solve_full(U, b[r], dims, KAPPA, MU, 0.0, n, apbc)[0]
        assert np.linalg.norm(s[r] - want) <= 16 * n * U16 * np.linalg.norm(want), r
        assert np.abs(s[r] - want).max() <= 64 * n * U16 * np.abs(want).max(), r


@pytest.mark.parametrize("dims,n_lp,n", [((12, 12, 12, 24), 9, 2), ((24, 12, 12, 24), 2, 1), ((16, 12, 12, 24), 2, 1)])
def test_estimates_on_larger_lattices(ctx, dims, n_lp, n):
    """LP solves of the loop estimators, 864 to 2592 tiles: the loops at every spatial
    momentum, transformed back, are eta^dag Gamma s at every site, |eta| = 1 per
    component.  So the density's error is at most sqrt(12) |ds| at a site: 16 n u
    sqrt(12) |s| normwise, 12 * 64 n u max |s| at every site."""
    U = S.gauge_field(dims, 0.3, 5)
    ctx.load_gauge(U, dims, KAPPA, MU)
    gam = [0, 5, 15]
    lp = tsm.stop(0.0, n, tsm.TSM_F16)
    got = ctx.loops(21, 4, 0, n_lp, tsm.stop(1e-8, 100, tsm.TSM_F32), lp, gam, None, batch=16, all_momenta=True)
    rho = np.fft.fftn(got["loops"], axes=(-3, -2, -1)) / (dims[0] * dims[1] * dims[2])
    gammas = gamma_list()
    want, norm, peak = 0, 0.0, 0.0
    for j in range(n_lp):
        eta = philox.noise(21, j, dims, 4)
        s = solver.solve_full(U, eta, dims, KAPPA, MU, 0.0, n)[0]
        want = want + np.stack([np.einsum('...rc,rs,...sc->...', eta.conj(), gammas[g], s) for g in gam]) / n_lp
        norm, peak = norm + np.linalg.norm(s) / n_lp, max(peak, np.abs(s).max())
    for g in range(len(gam)):
        assert np.linalg.norm(rho[g] - want[g]) <= 16 * n * U16 * np.sqrt(12) * norm, g
        assert np.abs(rho[g] - want[g]).max() <= 12 * 64 * n * U16 * peak, g
        print("gamma %d: error %.3e of the density's norm, worst site %.3e" % (
            gam[g], np.linalg.norm(rho[g] - want[g]) / np.linalg.norm(want[g]), np.abs(rho[g] - want[g]).max()))


@pytest.mark.parametrize("prec", [tsm.TSM_F16, tsm.TSM_BF16])
def test_production_lattice_residual(ctx, prec):
    """24^3x48, stopped at 5e-3 of the normal residual: the true residual, in FP64, is
    within 20 times that, the bound used on the small lattices."""
    dims = (24, 24, 24, 48)
    ctx.load_gauge(S.gauge_field(dims, 0.25, 3), dims, 0.1245, 0.005)
    b = philox.noise(1000, 0, dims, 4)
    _, iters, tres, st = ctx.solve(b, tsm.stop(5e-3, 60, prec))
    assert st == 0 and 0 < iters[0] < 60 and tres[0] < 20 * 5e-3
