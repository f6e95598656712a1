"""rsqrt64 (common.cuh), the FP64 path's 1/sqrt, against extended precision on the host.

One third-order Householder step from an estimate y0 good to 2^-20: with |h| <= 2^-19 the series remainder
5 |h|^3 / 16 is below 2^-58, the rounding of x y0 enters h as 2^-53 and the result as 2^-54, and the last
FMA rounds by 2^-53, so the relative error is below 1.51 x 2^-53.  Without the step's last term it would
be 1.4e-12.  Outside the normal range the plain expression's value is returned, bit for bit.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()


def _rsqrt(x):
    from paper_2409_04215_gb300.api import selftest_rsqrt64

    return selftest_rsqrt64(torch.tensor(x, device="cuda")).cpu().numpy()


@pytest.mark.parametrize("exponents", [(0, 2), (-40, 40), (-1022, 1024)])
def test_relative_error(exponents):
    rng = np.random.default_rng(1)
    n = 1 << 20
    mant = np.concatenate([1.0 + rng.random(n), 1.0 + np.arange(4096) / 4096.0, 2.0 - np.arange(1, 4097) * 2.0**-52,
                           1.0 + np.arange(4096) * 2.0**-52])
    x = np.ldexp(mant, rng.integers(exponents[0], exponents[1], mant.size))
    wide = np.longdouble
    assert np.finfo(wide).nmant >= 63
    exact = 1 / np.sqrt(x.astype(wide))
    err = np.abs(_rsqrt(x).astype(wide) / exact - 1)
    assert float(err.max()) <= 1.51 * 2.0**-53


def test_ends_of_the_normal_range_and_beyond():
    tiny, big = np.finfo(np.float64).tiny, np.finfo(np.float64).max
    ends = np.array([tiny, np.nextafter(tiny, 1.0), big, np.nextafter(big, 0.0)])
    exact = 1 / np.sqrt(ends.astype(np.longdouble))
    assert float(np.abs(_rsqrt(ends) / exact - 1).max()) <= 1.51 * 2.0**-53
    odd = np.array([0.0, -0.0, 5e-324, 1e-310, np.nextafter(tiny, 0.0), np.inf, -np.inf, np.nan, -1.0, -tiny, -5e-324])
    with np.errstate(all="ignore"):
        want = 1.0 / np.sqrt(odd)
    got = _rsqrt(odd)
    assert np.array_equal(got, want, equal_nan=True) and np.array_equal(np.signbit(got[:2]), np.signbit(want[:2]))
