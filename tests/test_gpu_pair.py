"""The FP64 reciprocal and the splitting into fp32 pairs of tcw_pair.cuh against exact
rationals, over the range that they handle by bits, its edges, and outside it."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2507_07816_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("pair") / "pair_check.so")
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", os.path.join(HERE, "pair_check.cu"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)

    def call(v):
        x = torch.as_tensor(np.asarray(v, np.float64), device="cuda:0")
        out = torch.empty((len(v), 4), dtype=torch.float64, device="cuda:0")
        torch.cuda.synchronize()
        assert lib.pair_check(ctypes.c_void_p(x.data_ptr()), len(v), ctypes.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy().T
    return call


def values():
    r = np.random.default_rng(7)
    m = np.concatenate([1 + r.random(3000), np.nextafter(2.0, 1.0) - 2.0 ** -52 * np.arange(20),
                        1 + 2.0 ** -24 * (1 + 2 * np.arange(20)),                 # halfway between floats
                        1 + 2.0 ** -24 * (1 + 2 * np.arange(20)) - 2.0 ** -52, 1 + 2.0 ** -23 * np.arange(20)])
    e = np.concatenate([r.integers(-60, 100, len(m) - 80), np.repeat([-60, 99, 0, 23], 20)])
    v = np.ldexp(m, e)
    return np.concatenate([v, -v])


def test_ordinary_range(check):
    """near_float: the nearest float, ties away from 0.  hi + lo: within 2^-48 of v (29 bits
    rounded to 24, below hi's last place).  Reciprocal: one rounding (2^-53 of 1/v) and
    the dropped terms, 2^-64."""
    v = values()
    near, hi, lo, rec = check(v)
    u = v.view(np.uint64)
    tie = (u & np.uint64((1 << 29) - 1)) == np.uint64(1 << 28)
    assert tie.sum() >= 40
    np.testing.assert_array_equal(near[~tie], v[~tie].astype(np.float32).astype(np.float64))
    assert np.all(np.abs(near[tie]) > np.abs(v[tie]))
    assert np.all(np.abs(near[tie] - v[tie]) == np.spacing(v[tie].astype(np.float32)).astype(np.float64).__abs__() / 2)
    np.testing.assert_array_equal(hi, near)
    for x, h, l, q in zip(v.tolist(), hi.tolist(), lo.tolist(), rec.tolist()):
        x, h, l, q = Fraction(x), Fraction(h), Fraction(l), Fraction(q)
        assert abs(x - h - l) <= abs(x) / 2 ** 48
        assert abs(q * x - 1) <= Fraction(1, 2 ** 53) + Fraction(1, 2 ** 64)


def test_outside_the_range(check):
    tiny, huge = 2.0 ** -60, 2.0 ** 100
    v = np.array([np.nextafter(tiny, 0), tiny, huge, np.nextafter(huge, 0), 2.0 ** -140, 3e-310, 2.0 ** 127, 1e300, 0.0,
                  np.inf, 1e-300])
    v = np.concatenate([v, -v, [np.nan]])
    near, hi, lo, rec = check(v)
    with np.errstate(all="ignore"):
        f = v.astype(np.float32)
        np.testing.assert_array_equal(near, f.astype(np.float64))
        np.testing.assert_array_equal(hi, f.astype(np.float64))
        np.testing.assert_array_equal(lo, (v - f.astype(np.float64)).astype(np.float32).astype(np.float64))
        inside = (np.abs(v) >= tiny) & (np.abs(v) < huge)
        np.testing.assert_array_equal(rec[~inside], (1.0 / v)[~inside])
        assert np.all(np.abs(rec[inside] * v[inside] - 1) <= 2.0 ** -52)
