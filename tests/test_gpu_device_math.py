"""The reciprocal and the FP64 exponential of the step against CUDA's own, in units in
the last place of the result.

vrcp: a correction whose rest is far below an ulp and one rounding at its end, so the
value is the correctly rounded one or its neighbour (1 ulp).  exp_neg_table: half an
ulp each from the table entry, the series and the last operation, 1.5 in all;
CUDA's exp and expm1 are within 1 ulp: 2.5, so at most 2 whole steps apart, 3 where a
power of two lies between.
"""
import ctypes

import numpy as np
import pytest

import launch_rules

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    return launch_rules.compile_so("device_math.cu")


def call(fn, x, *extra):
    got, want = np.empty_like(x), np.empty_like(x)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert fn(p(x), p(got), p(want), len(x), *extra) == 0
    return got, want


def steps_apart(a, b):
    i = np.int64 if a.dtype == np.float64 else np.int32
    return np.abs(a.view(i).astype(np.int64) - b.view(i).astype(np.int64))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_reciprocal(lib, dtype):
    rng = np.random.default_rng(1)
    tops = np.float64(2.0) ** np.arange(-60, 61)
    x = np.concatenate([rng.uniform(0.02, 12.0, 1 << 20), 2.0 ** rng.uniform(-60, 60, 1 << 18), tops,
                        np.nextafter(tops.astype(dtype), dtype(0)), np.nextafter(tops.astype(dtype), dtype(np.inf))])
    x = np.concatenate([x, -x]).astype(dtype)
    got, want = call(lib.run_rcp32 if dtype == np.float32 else lib.run_rcp64, x)
    assert steps_apart(got, want).max() <= 1


@pytest.mark.parametrize("one_minus", [0, 1])
def test_exponential(lib, one_minus):
    rng = np.random.default_rng(2)
    grid = np.concatenate([np.arange(1, 512) / 64.0, (np.arange(1, 511) + 0.5) / 64.0])
    x = np.concatenate([rng.uniform(2.0 ** -6, 7.9921875, 1 << 20), grid, np.nextafter(grid, 0), np.nextafter(grid, 9),
                        [np.nextafter(7.9921875, 0)]])
    x = x[(x >= 2.0 ** -6) & (x < 7.9921875)]
    assert x.min() == 2.0 ** -6 and x.max() == np.nextafter(7.9921875, 0)
    got, want = call(lib.run_exp64, x, one_minus)
    assert (got > 0).all()               # every one of them takes the table
    assert steps_apart(got, want).max() <= 3
    outside = np.array([np.nextafter(2.0 ** -6, 0), 7.9921875, -1.0, 0.0, np.inf, -np.inf, np.nan])
    assert (call(lib.run_exp64, outside, one_minus)[0] == -1.0).all()
