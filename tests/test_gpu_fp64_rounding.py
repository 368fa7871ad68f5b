"""The rounding claimed for the stage kernels' integer reciprocal (within 0.504 units in the last place) and square
root (correctly rounded), at arguments where the last step decides: mantissas next to 1 and 2, next to powers of 4,
and squares of numbers half-way between two doubles. Reference: extended precision (numpy.longdouble, at least 64 bits:
the error of the reference is below 2^-11 units)."""
import numpy as np
import pytest
import torch

from paper_1912_12059_gb300 import nsk

pytestmark = pytest.mark.gpu


def _eval(gpu, fn, x):
    xt = torch.from_numpy(x).to(gpu)
    y = torch.empty_like(xt)
    nsk._test_hook_math(fn, xt, y)
    torch.cuda.synchronize()
    return y.cpu().numpy()


def _arguments():
    g = np.random.Generator(np.random.PCG64(11))
    near = np.concatenate([1.0 + np.arange(2000) * 2.0**-52, 2.0 - np.arange(1, 2000) * 2.0**-52])
    x = np.concatenate([np.ldexp(g.uniform(1.0, 2.0, 500000), g.integers(-118, 118, 500000)),
                        np.concatenate([near * 4.0**k for k in (-50, -1, 0, 1, 2, 50)]), near * 0.5, near * 2.0])
    # the doubles around the squares of half-way points between neighbouring roots
    s = np.ldexp(g.uniform(1.0, 2.0, 200000), g.integers(-50, 50, 200000))
    mid = s.astype(np.longdouble) + 0.5 * np.spacing(s)
    sq = (mid * mid).astype(np.float64)
    return np.concatenate([x, sq, np.nextafter(sq, 0.0), np.nextafter(sq, np.inf)])


def test_reciprocal_within_its_bound(gpu):
    x = _arguments()
    r = _eval(gpu, 0, x)
    ex = 1.0 / x.astype(np.longdouble)
    ulp = np.spacing(ex.astype(np.float64))
    err = np.abs(r - ex) / ulp
    assert err.max() <= 0.505, (float(err.max()), x[err.argmax()])


def test_square_root_correctly_rounded(gpu):
    x = _arguments()
    assert np.array_equal(_eval(gpu, 1, x), np.sqrt(x))
