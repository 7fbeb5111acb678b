"""Rounding of the stencils, at fields where it can be told apart exactly."""
import numpy as np
import pytest

from oracle import dirac
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu


def _unit_gauge(dims):
    U = np.zeros(S.gauge_field(dims, 0.3, 1).shape, dtype=np.complex128)
    U[...] = np.eye(3)
    return U


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (12, 12, 12, 12)])
@pytest.mark.parametrize("mu", [0, 1, 2, 3])
@pytest.mark.parametrize("dagger", [False, True])
def test_fp64_hops_of_a_direction_round_once(ctx, dims, mu, dagger):
    """Unit links, one component 1 at x + mu and 2^-53 at x - mu: the lower
    components of site x are their difference times a unit, 1 - 2^-53, which FP64
    holds exactly; formed as 2 * 1 - (1 + 2^-53) it would be 1.  kappa = 1 and mu
    = 0, so that D applies H without another rounding (both FP64 kernels of D)."""
    U = _unit_gauge(dims)
    ctx.load_gauge(U, dims, 1.0, 0.0, antiperiodic_t=False)
    a = np.zeros(S.random_spinor(dims, 1).shape, dtype=np.complex128)
    b = np.zeros_like(a)
    x = [2, 2, 2, 2]
    for f, step, value in ((a, 1, 1.0), (b, -1, 2.0 ** -53)):
        y = list(x)
        y[mu] += step
        f[y[3], y[2], y[1], y[0], 0, 1] = value
    hops = [dirac.hop(U, f, dims, antiperiodic_t=False, adjoint=dagger) for f in (a, b)]
    want = (a + b) - (hops[0] + hops[1])   # every sum has at most two terms: one rounding
    assert np.any(np.abs(want) == 1 - 2.0 ** -53)
    got = ctx.dslash(a + b, tsm.TM_OP_FULL, dagger, tsm.TSM_F64)
    assert np.array_equal(got, want)
