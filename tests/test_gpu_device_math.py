"""Device functions of the kernels against 64-bit values, compiled from the
kernels' own headers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -23  # of a result in [1, 2): relative errors below count these


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2504_18583_gb300 import _build
    out = str(tmp_path_factory.mktemp("math") / "device_math.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-I" + _build.CSRC, "-shared", "-o", out,
                    os.path.join(ROOT, "tests", "device_math.cu")], check=True)
    return ctypes.CDLL(out)


def apply(f, *args):
    import torch
    dev = [torch.as_tensor(a, dtype=torch.float32, device="cuda") for a in args]
    y = torch.empty_like(dev[0])
    assert f(*[ctypes.c_void_p(t.data_ptr()) for t in dev], ctypes.c_void_p(y.data_ptr()), y.numel()) == 0
    return y.cpu().numpy().astype(np.float64)


def test_silu_is_a_few_ulp_over_its_range(lib):
    """z / (1 + e^-z): the exponential is within 2 ulp, the sum and the
    quotient round once each (at most half an ulp), and a result's ulp is up
    to twice as coarse as the factor's: 2 + 2 x 0.5, doubled at most, is 6."""
    z = np.concatenate([np.linspace(-80, 80, 200_001), np.linspace(-2, 2, 50_001)]).astype(np.float32)
    got = apply(lib.device_silu, z)
    want = z.astype(np.float64) / (1.0 + np.exp(-z.astype(np.float64)))
    rel = np.abs(got - want)[want != 0] / np.abs(want)[want != 0]
    print("largest error, ulp", rel.max() / ULP)
    assert rel.max() <= 6 * ULP
    assert apply(lib.device_silu, np.float32([0.0, -200.0, 200.0])).tolist() == [0.0, -0.0, 200.0]
