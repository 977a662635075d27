"""FP64 helpers of the rotation and the training's row stage (dsmc_selftest_math) against the value in more than
64 bits (numpy's long double) and against CUDA's own routines.

Bounds, from the operations: a reciprocal square root or square root ends in one rounding (2^-53), the rounding of
its first product counts half, and the series is cut at 2^-55: below 2^-52 in all.  Sine and cosine end in one
rounding of a value below 1 (2^-54), take the table's value (2^-53) and products below 2^-5 of it: below 2^-52.
"""
import numpy as np
import pytest

from gpu_util import ctx, cuda, host

pytestmark = pytest.mark.gpu

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288419716939937510")


def _f(which, x):
    out = host(ctx().selftest_math(which, cuda(x)))
    assert ctx().sync_status() == 0
    return out


def _arguments(lo, hi, rng):
    """Positive values over 2^lo .. 2^hi, all mantissas at ordinary exponents, and next to powers of two."""
    p = np.exp2(np.arange(lo, hi, dtype=np.float64))
    return np.concatenate([np.exp2(rng.uniform(lo, hi, 400000)), np.exp2(rng.uniform(-4, 4, 400000)), p,
                           np.nextafter(p, np.inf), np.nextafter(p[1:], 0.0)])


@pytest.mark.parametrize("own,cuda_own,exact", [(4, 5, lambda x: 1 / np.sqrt(x)), (6, 7, np.sqrt)])
def test_square_roots(own, cuda_own, exact):
    x = _arguments(-930, 930, np.random.default_rng(1))
    want = exact(x.astype(LD))
    err = np.abs(_f(own, x) / want - 1)
    assert err.max() <= 2.0 ** -52, float(np.log2(err.max()))
    # and over the same range CUDA's own routine within its documented 1 ulp: the two differ by that and the bound
    ref = _f(cuda_own, x)
    assert (np.abs(_f(own, x) - ref) <= 2 * np.spacing(ref)).all()


@pytest.mark.parametrize("own,cuda_own", [(4, 5), (6, 7)])
def test_square_roots_outside_the_plain_range_are_cudas(own, cuda_own):
    edge = np.exp2(930.0)
    x = np.concatenate([np.exp2(np.random.default_rng(2).uniform(930, 1023, 10000)), [edge, np.finfo(np.float64).max, np.inf],
                        np.exp2(np.random.default_rng(3).uniform(-1074, -930.001, 10000)), [0.0, -0.0, -1.0, np.nan, 5e-324]])
    assert np.array_equal(_f(own, x), _f(cuda_own, x), equal_nan=True)


@pytest.mark.parametrize("own,cuda_own,exact", [(8, 9, np.sin), (10, 11, np.cos)])
def test_sine_and_cosine_of_an_fp32_angle(own, cuda_own, exact):
    rng = np.random.default_rng(4)
    step = np.pi / 256
    x = np.concatenate([rng.uniform(-np.pi, np.pi, 400000), rng.uniform(-4096, 4096, 400000), 10.0 ** rng.uniform(-40, 0, 50000),
                        np.arange(-600, 600) * step, [0.0, -0.0, 4095.9998, -4095.9998]]).astype(np.float32).astype(np.float64)
    got = _f(own, x)
    err = np.abs(got - exact(x.astype(LD)))
    assert err.max() <= 2.0 ** -52, float(np.log2(err.max()))
    far = np.concatenate([[4096.0, -4096.0, 1e6, -3e38, np.inf, np.nan], rng.uniform(4096, 1e5, 1000)])
    assert np.array_equal(_f(own, far), _f(cuda_own, far), equal_nan=True)
    assert np.abs(got - _f(cuda_own, x)).max() <= 2.0 ** -51   # sincos: 1 ulp of a value below 1


@pytest.mark.parametrize("own,cuda_own,exact", [(12, 13, np.sin), (14, 15, np.cos)])
def test_sine_and_cosine_of_a_uniform_turn(own, cuda_own, exact):
    rng = np.random.default_rng(5)
    k = np.concatenate([rng.integers(0, 1 << 53, 800000), np.arange(512, dtype=np.int64) << 44,
                        (np.arange(1, 512, dtype=np.int64) << 44) - 1, [0, 1, (1 << 53) - 1]])
    x = k.astype(np.float64) * 2.0 ** -53
    got = _f(own, x)
    err = np.abs(got - exact(2 * PI * x.astype(LD)))
    assert err.max() <= 2.0 ** -52, float(np.log2(err.max()))
    assert np.abs(got - _f(cuda_own, x)).max() <= 2.0 ** -51


def test_selftest_math_refuses_other_functions():
    from paper_2602_21244_gb300 import dsmc as D
    for which in (-1, 16):
        with pytest.raises(D.DsmcError):
            ctx().selftest_math(which, cuda(np.ones(1)))
