"""Stopping rule of the solves at the ends of the FP64 range."""
import numpy as np
import pytest

from oracle import solver
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

KAPPA, MU = 0.124, 0.01


@pytest.mark.parametrize("scale,tol,err", [(1e-154, 1e-10, 1e-5), (1e-156, 1e-10, 1e-5), (1e-140, 1e-10, 1e-9), (1e140, 1e-10, 1e-9)])
def test_scaled_sources_converge(ctx, scale, tol, err):
    """D is linear: the solution scales with the source.  At 1e-154 the squared
    residual underflows to zero at a relative residual of about 1e-8 (components of
    1e-162), with tol^2 |r0|^2 = 0: the rule is met there, as it is on the norms
    themselves.  (Some scales below 1e-154 stagnate in either form: alpha and beta
    are ratios of subnormals.)  err: 1 / |D^-1| is of order 0.1, so ten to a hundred times the
    residual reached."""
    dims = (4, 4, 4, 4)
    U = S.gauge_field(dims, 0.3, 71)
    ctx.load_gauge(U, dims, KAPPA, MU)
    b = S.random_spinor(dims, 72)
    want = solver.solve_full(U, b, dims, KAPPA, MU, 1e-13, 5000)[0]
    s, iters, _, st = ctx.solve(scale * b, tsm.stop(tol, 500, tsm.TSM_F64))
    assert st == 0 and 0 < iters[0] < 500
    assert np.linalg.norm(s / scale - want) <= err * np.linalg.norm(want)
