"""FP16 solves of tm_solve_batch on either side of the line between the grouped
tensor-core stencil (8 sources at a time) and plain fields.

The line is 108 sites per SM, 16416 on 152 SMs, whatever the batch.  Bounds of the
truncated solves: those derived in test_gpu_mma_hop.py, 16 n u normwise and 64
n u of the largest component (n iterations, u = 2^-11).
"""
import numpy as np
import pytest

from oracle import solver
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

KAPPA, MU, U16, N = 0.124, 0.01, 2.0 ** -11, 2


@pytest.mark.parametrize("dims,nrhs,apbc", [
    ((8, 12, 10, 18), 3, True), ((6, 14, 10, 20), 2, False), ((10, 10, 14, 12), 1, True), ((18, 10, 10, 10), 9, True)])
def test_truncated_solves_of_both_routes(ctx, dims, nrhs, apbc):
    """17280, 16800, 16800 and 18000 sites: plain fields, odd row lengths; the same
    call on the first 8 timeslices' lattice runs grouped."""
    for d in (dims, dims[:3] + (8,)):
        U = S.gauge_field(d, 0.3, 5)
        ctx.load_gauge(U, d, KAPPA, MU, antiperiodic_t=apbc)
        b = S.random_spinor(d, 6, batch=(nrhs,))
        s, iters, _, _ = ctx.solve(b, tsm.stop(0.0, N, tsm.TSM_F16))
        assert np.all(iters == N)
        for r in {0, nrhs - 1}:
            want = solver.solve_full(U, b[r], d, KAPPA, MU, 0.0, N, apbc)[0]
            assert np.linalg.norm(s[r] - want) <= 16 * N * U16 * np.linalg.norm(want), (d, r)
            assert np.abs(s[r] - want).max() <= 64 * N * U16 * np.abs(want).max(), (d, r)


@pytest.mark.parametrize("dims", [(8, 8, 16, 16), (8, 8, 16, 18)])
def test_a_source_does_not_depend_on_its_batch(ctx, dims):
    """16384 and 18432 sites, just below and above the line; sources that stop at
    different iterations, every link-sharing block shape."""
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, KAPPA, MU)
    b = S.random_spinor(dims, 8, batch=(11,))
    b[4] *= 1e-2
    b[6] = 0.0
    stop = tsm.stop(5e-3, 60, tsm.TSM_F16)
    s, iters, _, _ = ctx.solve(b, stop)
    for sources, regs in tsm.TILE_SHAPES:
        tsm.tsm_set_tile(ctx.h, tsm.TSM_F16, sources, regs)
        for r in (0, 4, 6, 10):
            one, it, _, _ = ctx.solve(b[r], stop)
            assert it[0] == iters[r] and np.array_equal(one, s[r]), (r, sources, regs)


def test_one_source_of_a_large_lattice_holds_one_source(libtsm):
    """A single FP16 solve at 16^3x32 allocates the fields of one source: 8 parity
    fields of 96 bytes and 5 of 48 bytes per half-site, 66 MB, and less than 2 MB of
    rounding for each of some 20 buffers.  A group of 8 would hold 110 MB more."""
    import torch
    dims = (16, 16, 16, 32)
    V = int(np.prod(dims))
    c = tsm.Context(0)
    try:
        c.load_gauge(S.gauge_field(dims, 0.3, 9), dims, KAPPA, MU)
        b = torch.from_numpy(S.random_spinor(dims, 10)).cuda()
        s = torch.empty_like(b)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        tsm.tm_solve_batch(c.h, b, s, tsm.stop(0.0, 2, tsm.TSM_F16), 1)
        used = free - torch.cuda.mem_get_info()[0]
        assert used <= V // 2 * (8 * 96 + 5 * 48) + 20 * (2 << 20), used
    finally:
        c.close()


def test_tuner_keeps_the_shape_of_plain_solves(ctx):
    """The estimators' FP16 solves have no block shape to tune; the one set for the
    solves on plain fields is reported and left as it is, first time and cached."""
    dims = (4, 4, 4, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, KAPPA, MU)
    stop = tsm.stop(0.0, 3, tsm.TSM_F16)
    for shape in ((4, 96), (8, 80)):
        tsm.tsm_set_tile(ctx.h, tsm.TSM_F16, *shape)
        for _ in range(2):
            width, sources, regs, times = tsm.tsm_tune(ctx.h, stop)
            assert (sources, regs) == shape and np.all(times > 0) and width in (8, 16, 32, 64)


HP, LP = tsm.stop(1e-10, 5000, tsm.TSM_F32, reliable=True), tsm.stop(5e-3, 60, tsm.TSM_F16)
GAM = list(range(16))


@pytest.mark.parametrize("kw", [{}, {"estimator": 1}, {"estimator": 2}, {"deriv_mask": 5}, {"hp_warm_start": True}])
@pytest.mark.parametrize("n_hp,n_lp,batch", [(1, 1, 1), (3, 2, 8), (3, 9, 2), (11, 20, 4), (8, 3, 8)])
def test_estimates_do_not_depend_on_shared_groups(ctx, kw, n_hp, n_lp, batch):
    """LP-set sources that share the HP set's last group of 8 have the values of a call
    without HP sources, the HP set's those of a call without LP sources."""
    dims = (4, 4, 2, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, KAPPA, MU)
    def run(hp, lp):
        return ctx.loops(9, 4, 0, 0, HP, LP, GAM, S.default_momenta(4), hp_range=hp, lp_range=lp, per_source=True,
                         batch=batch, **kw)
    both = run((0, n_hp), (n_hp, n_hp + n_lp))
    hp_only, lp_only = run((0, n_hp), (n_hp, n_hp)), run((0, 0), (n_hp, n_hp + n_lp))
    assert np.array_equal(both["per_corr"], hp_only["per_corr"])
    assert np.array_equal(both["per_lp"], lp_only["per_lp"])
    assert both["stats"]["lp_iters"] == hp_only["stats"]["lp_iters"] + lp_only["stats"]["lp_iters"]
    comb = ctx.combine(both["per_corr"], both["per_lp"])
    assert np.array_equal(comb["loops"], both["loops"]) and np.array_equal(comb["err"], both["err"])


@pytest.mark.parametrize("n_hp,n_lp", [(2, 9), (9, 40)])
def test_all_momenta_with_shared_groups(ctx, n_hp, n_lp):
    """The running moments of both sets against the direct projection (bounds of
    test_gpu_fft.py's mixed tier)."""
    dims = (4, 6, 2, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 5), dims, KAPPA, MU)
    moms = [(0, 0, 0), (1, 0, 0), (-1, 2, 1)]
    direct = ctx.loops(13, 4, n_hp, n_lp, HP, LP, GAM, moms, batch=4)
    allq = ctx.loops(13, 4, n_hp, n_lp, HP, LP, GAM, None, batch=4, all_momenta=True)
    for k, (nx, ny, nz) in enumerate(moms):
        i = (slice(None), slice(None), nz % dims[2], ny % dims[1], nx % dims[0])
        for name, tol in (("loops", 1e-5), ("err", 1e-4)):
            scale = np.abs(direct[name][:, k, :]).max()
            assert np.abs(allq[name][i] - direct[name][:, k, :]).max() < tol * scale, name


def test_few_lp_sources_share_the_group_of_the_hp_set(ctx):
    """1 HP source and up to 7 LP sources are one group: LP sources add no solve, a few
    launches for their noise and contraction."""
    dims = (4, 4, 4, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, KAPPA, MU)
    fixed = tsm.stop(0.0, 8, tsm.TSM_F16)
    def launches(n_lp):
        a = tsm.tsm_launch_count(ctx.h)
        ctx.loops(9, 4, 1, n_lp, HP, fixed, GAM, S.default_momenta(4), batch=8)
        return tsm.tsm_launch_count(ctx.h) - a
    base = launches(0)
    assert launches(1) <= base + 6 and launches(7) <= base + 6
