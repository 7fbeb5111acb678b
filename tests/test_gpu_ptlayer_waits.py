"""Shared memory and waits of the fused network layer."""
import numpy as np
import pytest

from oracle import ptnet
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -9


@pytest.mark.parametrize("channels,dims", [([1, 9, 16, 1], (8, 6, 10, 12)), ([1, 32, 2, 1], (6, 14, 10, 6))])
def test_weights_survive_the_zero_fill(ctx, channels, dims):
    """The start of a block zeroes the activations' part of both stages while the
    first weights arrive beside it: 200 passes give the same bits, with other
    kernels' data left in shared memory between them, and the oracle's values
    (4 L u normwise)."""
    U = S.gauge_field(dims, 0.3, 3)
    ctx.load_gauge(U, dims, 0.124, 0.01)
    net = tsm.Network(channels, seed=1, init_scale=1.0)
    L = len(channels) - 1
    ws = [net.get_weights(l) for l in range(L)]
    x = S.random_spinor(dims, 5, batch=(1, 1))
    y = net.forward(ctx, x)
    want = ptnet.net_forward(U, ws, x[0], dims)[-1]
    assert np.linalg.norm(y[0] - want) <= 4 * L * U_BF16 * np.linalg.norm(want)
    for k in range(200):
        if k % 10 == 0:
            ctx.dslash(x[0, 0], tsm.TM_OP_FULL, False, tsm.TSM_F64)
        assert np.array_equal(net.forward(ctx, x), y), k

TIMEOUT = -6   # TSM_ERR_TIMEOUT


def _timeout_and_recovery(ctx, channels, dims):
    U = S.gauge_field(dims, 0.3, 3)
    ctx.load_gauge(U, dims, 0.124, 0.01)
    net = tsm.Network(channels, seed=1, init_scale=1.0)
    x = S.random_spinor(dims, 5, batch=(1, 1))
    y = net.forward(ctx, x)
    tsm.tsm_umma_inject_timeout(True)
    try:
        with pytest.raises(tsm.TsmError) as e:
            net.forward(ctx, x)
        assert e.value.status == TIMEOUT
    finally:
        tsm.tsm_umma_inject_timeout(False)
    assert np.array_equal(net.forward(ctx, x), y)


def test_timeout_of_the_gemm_is_reported_once(ctx):
    """Operand copies withheld on the host's request (nothing is in flight, every
    wait ends): the call on a lattice of few blocks, gather and GEMM, reports
    TSM_ERR_TIMEOUT and the next one computes again."""
    _timeout_and_recovery(ctx, [1, 5, 1], (4, 4, 4, 4))


@pytest.mark.parametrize("channels", [[1, 5, 1], [1, 24, 17, 1]])
def test_timeout_of_the_fused_layer(ctx, channels):
    """The same on a lattice of 138 blocks of the fused layer, one and two blocks
    per SM: the first stage's weights never come, every thread leaves the loop at
    that stage, tensor memory is freed."""
    _timeout_and_recovery(ctx, channels, (8, 6, 10, 12))
