"""rcp3 and sqrt3 (csrc/lbm_phase.cuh) against the correctly rounded quotient and root."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rcp_sqrt(tmp_path_factory):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1512_01977_gb300 import build

    so = str(tmp_path_factory.mktemp("math") / "libdevice_math.so")
    cmd = [build.NVCC, *build.ARCH, *build.FLAGS, "-shared", "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
           os.path.join(ROOT, "tests", "device_math.cu"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(so).rcp_sqrt

    def call(x):
        d = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        out = torch.empty((2, x.size), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert f(ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(out[0].data_ptr()), ctypes.c_void_p(out[1].data_ptr()),
                 x.size) == 0
        return out.cpu().numpy()

    return call


@pytest.mark.parametrize("lo,hi", [(-1, 1), (-12, 3), (-300, 300)])
def test_rounding(rcp_sqrt, lo, hi):
    """Within a unit in the last place, and correctly rounded but where the exact value lies that close to the
    middle between two numbers: the hardware's approximations are good to 2^-19.9, the series leave out terms of
    2^-59.7 (reciprocal) and 2^-59.4 (root), so at most 2 x 2^-6.4 of the values, 2.4 per cent."""
    rng = np.random.default_rng(1)
    x = 10.0 ** rng.uniform(lo, hi, 1 << 20)
    r, s = rcp_sqrt(x)
    for got, want in ((r, 1.0 / x), (s, np.sqrt(x))):
        assert np.all(np.abs(got - want) <= np.spacing(want))
        assert np.mean(got != want) <= 0.024


def test_special_values(rcp_sqrt):
    """What the division and the root give for zeros, subnormal values and results, infinities and NaN (the root: 0 for
    what is not positive)."""
    tiny, big = np.finfo(float).tiny, np.finfo(float).max
    x = np.array([0.0, np.inf, np.nan, 5e-324, 1e-310, np.nextafter(tiny, 0), tiny, np.nextafter(tiny, 1), 2.0 ** 1021,
                  np.nextafter(2.0 ** 1021, 0), 2.0 ** 1022, 1.5 * 2.0 ** 1022, 2.0 ** 1023, big])
    x = np.concatenate([x, -x])
    r, s = rcp_sqrt(x)
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(r, 1.0 / x)
        np.testing.assert_array_equal(s, np.where(x > 0, np.sqrt(x), 0.0))
