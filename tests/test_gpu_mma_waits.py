"""The bounded ring waits of the tensor-core stencil run out on stages that nothing
fills (copies withheld on the host's request, nothing in flight): the call
reports TSM_ERR_TIMEOUT, and the next one on the same context has the bits of an
undisturbed one."""
import numpy as np
import pytest

from paper_1211_0126_gb300 import synthetic as S
from paper_1211_0126_gb300 import tsm

pytestmark = pytest.mark.gpu

TIMEOUT = -6   # TSM_ERR_TIMEOUT


def _fails_then_recovers(call, same):
    want = call()
    tsm.tsm_umma_inject_timeout(True)
    try:
        with pytest.raises(tsm.TsmError) as e:
            call()
        assert e.value.status == TIMEOUT
    finally:
        tsm.tsm_umma_inject_timeout(False)
    assert same(call(), want)


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (12, 4, 4, 8)])
def test_solves_report_and_recover(ctx, dims):
    """Tiles of 4 and of 6 half-sites; a part-filled second group."""
    ctx.load_gauge(S.gauge_field(dims, 0.3, 3), dims, 0.124, 0.01)
    b = S.random_spinor(dims, 4, batch=(9,))
    _fails_then_recovers(lambda: ctx.solve(b, tsm.stop(5e-3, 60, tsm.TSM_F16))[0], np.array_equal)


def test_estimates_and_tuner_report_and_recover(ctx):
    dims = (4, 4, 4, 4)
    ctx.load_gauge(S.gauge_field(dims, 0.3, 3), dims, 0.124, 0.01)
    hp, lp = tsm.stop(1e-10, 5000, tsm.TSM_F32, reliable=True), tsm.stop(5e-3, 60, tsm.TSM_F16)
    _fails_then_recovers(lambda: ctx.loops(5, 4, 2, 9, hp, lp, list(range(16)), S.default_momenta(4))["loops"],
                         np.array_equal)
    _fails_then_recovers(lambda: tsm.tsm_tune(ctx.h, tsm.stop(0.0, 3, tsm.TSM_F16))[3].shape, lambda a, b: a == b)
