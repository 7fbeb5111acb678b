"""Rounding of the kernels' three-term complex products against 64 bits: two chains of
three multiply-adds and an addition may not be further off than the sum of three
separately formed products.  rms values over N independent errors scatter by
1 / sqrt(N) relative to each other; three times that is allowed."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1211_0126_gb300 import build
from paper_1211_0126_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("dot3") / "dot3_rounding.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "dot3_rounding.cu")
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", out, src, "-lcudart"] +
                   build._rpath(), check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("kind", ["random", "links", "links near the identity"])
def test_error_no_larger_than_that_of_summed_products(lib, kind):
    """a: random numbers, or rows of SU(3) links with large (eps = 3) or small (0.25)
    angles; b: random numbers.  conj(a) b has the errors of a b with other signs."""
    import torch
    n = 3 << 17
    rng = np.random.default_rng(3)
    if kind == "random":
        a = rng.standard_normal((n, 3, 2))
    else:
        U = S.random_su3(rng, (n // 3,), 3.0 if kind == "links" else 0.25)
        a = np.stack([U.real, U.imag], -1).reshape(n, 3, 2)
    b = rng.standard_normal((n, 3, 2))
    a, b = (torch.from_numpy(x.astype(np.float32)).cuda() for x in (a, b))
    out = [torch.full((n, 2), float("nan"), device="cuda") for _ in range(4)]
    torch.cuda.synchronize()
    assert lib.dot3_rounding(*[ctypes.c_void_p(x.data_ptr()) for x in [a, b] + out], n) == 0
    ad, bd = (torch.view_as_complex(x.double()) for x in (a, b))
    for conj, k in ((False, 0), (True, 2)):
        ref = torch.view_as_real(((ad.conj() if conj else ad) * bd).sum(1))
        plain = torch.view_as_real((ad * bd).sum(1))
        err = ((out[k].double() - ref) ** 2).mean().sqrt().item()
        err_sums = ((out[3].double() - plain) ** 2).mean().sqrt().item()
        chain = ((out[1].double() - plain) ** 2).mean().sqrt().item()
        print("%s, %s: ratio %.4f (one chain %.4f)" % (kind, "conj(a) b" if conj else "a b", err / err_sums, chain / err_sums))
        assert err <= err_sums * (1 + 3 / np.sqrt(ref.numel()))
