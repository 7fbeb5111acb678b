"""Canonical input and output of the operators at the edges of their kernels.

Fields enter and leave through blocks of 128 lexicographic sites (sizes below:
one partial block, an exact one, several with a remainder), and D_tm in FP64
runs four threads per site below 19456 sites and one above: both sides of that
line against the oracle, with both daggers.  Bounds: those of the operator in
each tier (1e-12, 1e-5, 5e-3 normwise).  Values that the narrowing to FP32
treats apart (zeros, subnormals, numbers that round across a binade) come
through the FP32 tier as numpy rounds them.
"""
import numpy as np
import pytest

from oracle import dirac
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

KAPPA, MU = 0.124, 0.01
BOUND = {tsm.TSM_F64: 1e-12, tsm.TSM_F32: 1e-5, tsm.TSM_BF16: 5e-3 * 2, tsm.TSM_F16: 5e-3}


@pytest.mark.parametrize("dims", [(2, 4, 6, 2), (4, 4, 4, 2), (6, 4, 2, 2), (10, 4, 6, 4)])
@pytest.mark.parametrize("prec", [tsm.TSM_F64, tsm.TSM_F32, tsm.TSM_BF16, tsm.TSM_F16])
def test_operators_on_partial_blocks(ctx, dims, prec):
    U = S.gauge_field(dims, 0.3, 3)
    ctx.load_gauge(U, dims, KAPPA, MU)
    psi = S.random_spinor(dims, 4)
    even, odd = dirac.even_mask(dims), dirac.odd_mask(dims)
    for op, want in ((tsm.TM_OP_FULL, dirac.dtm(U, psi, dims, KAPPA, MU)),
                     (tsm.TM_OP_HOP_EO, dirac.hop(U, psi * odd, dims) * even),
                     (tsm.TM_OP_HOP_OE, dirac.hop(U, psi * even, dims) * odd)):
        got = ctx.dslash(psi, op, False, prec)
        assert np.linalg.norm(got - want) <= BOUND[prec] * np.linalg.norm(want), op
        if op != tsm.TM_OP_FULL:
            assert np.all((got * (odd if op == tsm.TM_OP_HOP_EO else even)) == 0)


@pytest.mark.parametrize("dims", [(8, 8, 8, 16), (12, 12, 12, 12)])
@pytest.mark.parametrize("dagger", [False, True])
def test_full_operator_fp64_both_kernels(ctx, dims, dagger):
    U = S.gauge_field(dims, 0.3, 5)
    ctx.load_gauge(U, dims, KAPPA, MU)
    psi = S.random_spinor(dims, 6)
    want = dirac.dtm(U, psi, dims, KAPPA, MU, adjoint=dagger)
    got = ctx.dslash(psi, tsm.TM_OP_FULL, dagger, tsm.TSM_F64)
    assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)


def test_narrowing_rounds_like_the_cast(ctx):
    """kappa = mu = 0: D is the identity, so the FP32 tier returns its rounded input."""
    dims = (4, 4, 4, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 7), dims, 0.0, 0.0)
    psi = S.random_spinor(dims, 8)
    flat = psi.reshape(-1).view(np.float64)
    special = [0.0, -0.0, 1e-40, -3e-42, 1e-50, 2.0 - 2.0 ** -30, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24,
               1.0 + 2.0 ** -24 + 2.0 ** -50, 2.0 ** -126, 2.0 ** -126 - 2.0 ** -151, -1.17549435e-38, 3.0e38]
    flat[:len(special)] = special
    got = ctx.dslash(psi, tsm.TM_OP_FULL, False, tsm.TSM_F32)
    want = flat.astype(np.float32).astype(np.float64)
    assert np.array_equal(got.reshape(-1).view(np.float64), want)
