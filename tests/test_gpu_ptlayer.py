"""The fused network layer at the edges of its tiles, against the oracle.

Channel counts whose (path, channel) groups leave a padded last stage (odd
counts, 9 and 27 groups), every tile width (16 to 256 columns) and the first
one past it (40 channels: the unfused kernels); volumes that leave a part-filled
last block of 42 sites, and one smaller than a block.  Bound: that of the
forward pass, 4 L u normwise with u = 2^-9 the BF16 unit roundoff.

(The fused kernel is taken from 120 blocks of 42 sites on: by the lattices of the
second test but its last.  Those of the first run the same layers through gather
and GEMM.)
"""
import numpy as np
import pytest

from oracle import ptnet
from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

U_BF16 = 2.0 ** -9


@pytest.mark.parametrize("channels,dims", [
    ([1, 1], (2, 2, 2, 2)), ([1, 2, 1], (4, 4, 2, 2)), ([1, 5, 1], (6, 4, 2, 2)), ([1, 9, 16, 1], (4, 2, 6, 4)),
    ([1, 24, 17, 1], (4, 4, 4, 2)), ([1, 32, 1], (4, 4, 2, 4)), ([1, 40, 1], (4, 2, 2, 4))])
def test_forward_matches_oracle(ctx, channels, dims):
    U = S.gauge_field(dims, 0.3, 3)
    ctx.load_gauge(U, dims, 0.124, 0.01)
    net = tsm.Network(channels, seed=1, init_scale=1.0)
    L = len(channels) - 1
    ws = [net.get_weights(l) for l in range(L)]
    x = S.random_spinor(dims, 5, batch=(2, 1))
    y = net.forward(ctx, x)
    for b in range(2):
        want = ptnet.net_forward(U, ws, x[b], dims)[-1]
        assert np.linalg.norm(y[b] - want) <= 4 * L * U_BF16 * np.linalg.norm(want)


@pytest.mark.parametrize("channels,dims", [
    ([1, 1], (8, 6, 10, 12)), ([1, 5, 2, 1], (6, 14, 10, 6)), ([1, 9, 16, 1], (8, 6, 10, 12)),
    ([1, 24, 17, 1], (8, 6, 10, 12)), ([1, 32, 1], (6, 14, 10, 6)), ([1, 40, 1], (8, 6, 10, 12)),
    ([1, 12, 1], (14, 10, 6, 6)), ([1, 12, 1], (6, 10, 14, 4))])
def test_fused_lattices_match_oracle(ctx, channels, dims):
    """The same at the fewest blocks (120) the fused kernel is taken for, with whole
    and part-filled last blocks, and just below.  Bound as above."""
    test_forward_matches_oracle(ctx, channels, dims)
