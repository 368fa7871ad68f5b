"""The stage kernels' quotients: FP64 from the integer reciprocal with a correction, FP32 as divided.

Bound (derived before any run): the reciprocal is within 0.504 units in the last place, its product with the
numerator within 1.6; the remainder x - q y is exact in one multiply-add, and its product with the reciprocal
is off by 2^-52 of the correction, so the corrected quotient is within 0.5 + 2^-50 units: 0.501 below.
"""
import numpy as np
import pytest
import torch

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


def _pairs():
    g = np.random.Generator(np.random.PCG64(5))
    n = 400000
    x = g.standard_normal(n) * 10.0 ** g.uniform(-30, 30, n)
    y = np.concatenate([10.0 ** g.uniform(-30, 30, n // 2), g.uniform(1e-3, 3.0, n // 2)])
    x[:1000] = 0.0
    return x, y


def test_fp64_quotients(gpu):
    x, y = _pairs()
    q = nsk._test_hook_div(torch.from_numpy(x).to(gpu), torch.from_numpy(y).to(gpu)).cpu().numpy()
    ex = x.astype(np.longdouble) / y.astype(np.longdouble)
    assert (np.abs(q - ex) <= 0.501 * np.spacing(np.abs(ex.astype(float)))).all()


def test_fp64_quotients_outside_the_domain(gpu):
    """CUDA's division decides for denominators outside (2^-120, 2^120), infinite quotients stay infinite."""
    x = np.array([1.0, -1.0, 0.0, np.inf, 3e300, 2.0, -3.0, np.nan, np.inf, -np.inf])
    y = np.array([0.0, 0.0, 0.0, 1e-200, 1e-200, 1e200, np.inf, 1.0, 1.5, 2.0])
    q = nsk._test_hook_div(torch.from_numpy(x).to(gpu), torch.from_numpy(y).to(gpu)).cpu().numpy()
    with np.errstate(all="ignore"):
        assert np.array_equal(q, x / y, equal_nan=True)


def test_fp32_quotients_are_divisions(gpu):
    g = np.random.Generator(np.random.PCG64(6))
    x, y = (g.uniform(0.1, 100.0, 400000).astype(np.float32) for _ in range(2))
    q = nsk._test_hook_div(torch.from_numpy(x.astype(float)).to(gpu), torch.from_numpy(y.astype(float)).to(gpu),
                           nsk.NSK_FP32_MIXED).cpu().numpy()
    assert np.array_equal(q.astype(np.float32), x / y)
