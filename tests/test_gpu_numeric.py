"""The stand-alone pieces of device arithmetic (csrc/numeric.cuh), compiled with
tests/unit_numeric.cu and compared bit for bit with the same operations in numpy, and the quotient
from a reciprocal with CUDA's division and numpy's."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    from paper_2012_15662_gb300 import build
    so = str(tmp_path_factory.mktemp("unit") / "libunit.so")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so,
                    os.path.join(HERE, "unit_numeric.cu"), "-lcudart"], check=True)
    return ctypes.CDLL(so)


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("terms", [1, 2, 7, 8, 9, 79, 158, 1000])
@pytest.mark.parametrize("signed", [False, True])
def test_running_sums_are_renormalised_double_float_sums(unit, terms, signed):
    n = 512
    rng = np.random.default_rng(terms)
    x = rng.standard_normal((terms, n))
    x *= x if not signed else 10.0 ** rng.integers(-6, 6, (terms, n))
    hi = x.astype(np.float32)
    lo = (x - hi).astype(np.float32)
    s, c = np.zeros(n, np.float32), np.zeros(n, np.float32)
    for ph, pl in zip(hi, lo):
        t = s + ph
        bb = t - s
        e = ((s - (t - bb)) + (ph - bb)) + (c + pl)
        s = t + e
        c = e - (s - t)
    out = [_dev(np.empty(n, np.float32)) for _ in range(2)]
    h, l = _dev(hi), _dev(lo)
    p = [ctypes.c_void_p(v.data_ptr()) for v in (h, l, *out)]
    assert unit.unit_df_sums(p[0], p[1], terms, n, p[2], p[3]) == 0
    np.testing.assert_array_equal(out[0].cpu().numpy(), s)
    np.testing.assert_array_equal(out[1].cpu().numpy(), c)


@pytest.mark.parametrize("lo,hi,near", [(1.0, 2.0, False), (1.9, 2.0, True), (1.999, 2.0, True), (1.0, 1.001, False)])
def test_quotient_is_the_division(unit, lo, hi, near):
    """Divisors over [lo, hi) and their last bits; dividends anywhere in [1, 2), or just below the
    divisor, where the first approximation is off by up to 1.5 ulp; scaled by powers of two."""
    n = 1 << 20
    rng = np.random.default_rng(int(1000 * lo))
    d = rng.uniform(lo, hi, n)
    d[:4096] = np.nextafter(hi, 0) - np.arange(4096) * 2.0**-52
    x = d * rng.uniform(0.94, 1.0, n) if near else rng.uniform(1.0, 2.0, n)
    x *= 2.0 ** rng.integers(-200, 200, n) * rng.choice([-1.0, 1.0], n)
    d *= 2.0 ** rng.integers(-100, 100, n)
    x[-1] = 0.0
    q, ref = _dev(np.empty(n)), _dev(np.empty(n))
    xd, dd = _dev(x), _dev(d)
    p = [ctypes.c_void_p(v.data_ptr()) for v in (xd, dd, q, ref)]
    assert unit.unit_quotients(p[0], p[1], n, p[2], p[3]) == 0
    np.testing.assert_array_equal(q.cpu().numpy(), ref.cpu().numpy())
    np.testing.assert_array_equal(ref.cpu().numpy(), x / d)
