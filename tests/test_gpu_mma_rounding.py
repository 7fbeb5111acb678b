"""Rounding of the tensor-core stencil against the FP32 multiply-adds it stands for.

Row 2 of a link is an FP16 pair there, and the tensor cores round sums towards
zero.  On the same FP16 fields and link rows the error of H psi against 64 bits
may be no larger than that of sums of FP32 products with row 2 in FP32.
"""
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
    out = str(tmp_path_factory.mktemp("mma") / "mma_rounding.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "mma_rounding.cu")
    subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-shared", "-o", out, src, "-lcudart"] +
                   build._rpath(), check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("eps", [0.25, 3.0])
def test_error_no_larger_than_that_of_fp32_products(lib, eps):
    """eps: links near the identity and far from it.  The ratio of two rms values
    over N independent errors scatters by 1 / sqrt(N); three times that is allowed."""
    import torch
    ns = 1 << 13
    rng = np.random.default_rng(5)
    fields = torch.from_numpy(rng.standard_normal((ns, 24, 24, 8)).astype(np.float16)).cuda()
    U = S.random_su3(rng, (ns, 8), eps)[..., :2, :]
    rows = torch.from_numpy(np.stack([U.real, U.imag], -1).astype(np.float16)).cuda()
    words = torch.zeros((ns, 8, 12), dtype=torch.int32, device="cuda")
    tc, f32 = (torch.full((ns, 8, 24), float("nan"), device="cuda") for _ in range(2))
    f64 = torch.full((ns, 8, 24), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.mma_rounding(*[ctypes.c_void_p(x.data_ptr()) for x in (fields, rows, words, tc, f32, f64)], ns) == 0
    e_tc, e_32 = (((x.double() - f64) ** 2).mean().sqrt().item() for x in (tc, f32))
    print("eps %g: tensor cores %.4e, FP32 products %.4e, ratio %.4f" % (eps, e_tc, e_32, e_tc / e_32))
    assert e_tc <= e_32 * (1 + 3 / np.sqrt(f64.numel()))
