"""The fixed-point sums of the CG iteration's kernels against exact sums.

A sum keeps 64 bits below the leading one of its largest summand and is rounded to FP64 once, so
it differs from the exact sum by at most half a unit in the last place of the result and, for each
summand cut (in its warp, and each warp's sum once more in the CTA's), one unit of the 64th bit.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2107_12371_gb300 import build as gbuild

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    torch.cuda.init()
    lib = str(tmp_path_factory.mktemp("fx") / "libfx_sums.so")
    subprocess.run([gbuild._nvcc()] + gbuild.NVCC_FLAGS +
                   ["-I", gbuild.CSRC, "-I", gbuild.INCLUDE, "-shared", "-o", lib,
                    os.path.join(HERE, "fx_sums.cu")], check=True)
    so = ctypes.CDLL(lib)

    def call(fn, a, *args, nout=1):
        out = np.empty(nout)
        assert fn(ctypes.c_void_p(a.ctypes.data), a.size, *args,
                  ctypes.c_void_p(out.ctypes.data)) == 0
        return out

    def fold(a, threads=None):
        threads = threads or max(64, -(-a.size // 32) * 32)
        fn = so.fx_fold64 if a.dtype == np.float64 else so.fx_fold32
        s, neg = call(fn, a, threads, nout=2)
        if not math.isfinite(s):
            assert math.isnan(s) and math.isnan(neg) or neg == -s
        else:
            # (within a sum's bound, not its negative: a warp's sum is cut towards minus infinity
            # where the CTA's warps are aligned)
            check(neg, -a)
        return s
    return fold, lambda a: call(so.fx_parts, a)[0]


def bound(a, exact):
    """Half a unit in the result's last place, and a unit of bit 64 per summand and warp."""
    top = max(abs(float(v)) for v in a)
    e = math.frexp(max(top, 2.0 ** -1022))[1] - 1  # top in [2^e, 2^(e + 1))
    cut = math.ldexp(1.0, e - 63) if e - 63 >= -1074 else 0.0
    # a warp's sum has its leading one up to eight bits above (1,024 summands: ten)
    return 0.5 * math.ulp(exact) + cut * (len(a) + 32 * 2 ** 10)


def check(got, a):
    exact = math.fsum(float(v) for v in a)
    assert abs(got - exact) <= bound(a, exact), (got, exact)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 160, 1000, 1024])
@pytest.mark.parametrize("spread", [0, 30, 70, 600])
def test_random_sums(fx, dtype, n, spread):
    """Mixed signs and magnitudes (2^-spread to 1; FP32 down to its denormals)."""
    rng = np.random.default_rng(n + spread)
    e = -rng.uniform(0, min(spread, 140 if dtype == np.float32 else spread), n)
    a = (rng.choice([-1, 1], n) * rng.uniform(1, 2, n) * 2.0 ** e).astype(dtype)
    check(fx[0](a), a)
    if dtype == np.float64 and n <= 160:
        check(fx[1](a), a)


@pytest.mark.parametrize("shift", [0, 1, 10, 21, 22, 31, 32, 33, 43, 44, 52, 53, 63])
def test_warps_of_unlike_magnitude(fx, shift):
    """Warp sums 2^shift apart are aligned by shifts below, at and above 32 bits; integers, so that
    sums of up to 64 bits are exact before the rounding."""
    a = np.ones(1024)
    a[:32] = 2.0 ** shift
    a[32:64] = -2.0 ** (shift // 2)
    check(fx[0](a), a)
    exact = 32 * 2 ** shift - 32 * 2 ** (shift // 2) + 960
    if exact < 2 ** 53:
        assert fx[0](a) == exact


@pytest.mark.parametrize("shift", [64, 65, 80, 200, 1000])
def test_summands_below_the_window_leave_no_trace(fx, shift):
    a = np.full(96, 2.0 ** -shift)
    a[40] = 1.0
    assert fx[0](a) == 1.0
    assert fx[0](a, 1024) == 1.0


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_exact_cancellation(fx, dtype):
    rng = np.random.default_rng(1)
    h = rng.standard_normal(512).astype(dtype)
    a = rng.permutation(np.concatenate([h, -h]))
    assert fx[0](a) == 0.0
    # one unit in the last place of the smallest summand is left (within 64 bits of the largest)
    h = (rng.integers(2 ** 20, 2 ** 21, 500)).astype(dtype)
    a = np.concatenate([h, -h, [1, 0]]).astype(dtype)
    assert fx[0](a) == 1.0
    # the parts' 160 values
    p = np.concatenate([h[:79], -h[:79], [3]]).astype(np.float64)
    assert fx[1](p) == 3.0


def test_round_to_nearest_even(fx):
    one = 2.0 ** 53
    for low, want in (([1.0], one), ([1.0, 0.25], one + 2), ([3.0], one + 4), ([2.0], one + 2),
                      ([-0.5], one), ([-1.0], one - 1), ([1.0, -0.25], one)):
        a = np.array([one] + low)
        assert fx[0](a) == want == math.fsum(a)
        assert fx[1](a) == want


def test_ends_of_the_exponent_range(fx):
    tiny, big = 5e-324, np.finfo(np.float64).max
    for a in ([tiny] * 3, [tiny, -tiny], [2.0 ** -1022, -tiny], [2.0 ** -1022, 2.0 ** -1022, -tiny],
              [2.0 ** -1021, -2.0 ** -1022, tiny], [big], [big, -big], [big, -big, tiny],
              [big / 2, big / 4], [2.0 ** 1023, -2.0 ** 1022]):
        a = np.array(a)
        check(fx[0](a), a)
        check(fx[1](a), a)
    assert fx[0](np.array([tiny] * 3)) == 3 * tiny
    assert fx[0](np.array([2.0 ** -1022, -tiny])) == 2.0 ** -1022 - tiny
    for a in ([big, big], [big] * 100, [2.0 ** 1023] * 2):
        assert fx[0](np.array(a)) == np.inf and fx[1](np.array(a)) == np.inf
    f = np.finfo(np.float32)
    a = np.array([f.max] * 64, np.float32)
    assert fx[0](a) == 64 * float(f.max)  # past FP32's range, not FP64's
    a = np.array([f.smallest_subnormal] * 33, np.float32)
    assert fx[0](a) == 33 * float(f.smallest_subnormal)
    a = np.array([f.tiny, -f.smallest_subnormal], np.float32)
    assert fx[0](a) == float(f.tiny) - float(f.smallest_subnormal)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("at", [0, 31, 500, 1023])
def test_what_is_not_finite_gives_nan(fx, dtype, bad, at):
    a = np.ones(1024, dtype)
    a[at] = bad
    assert math.isnan(fx[0](a))
    if dtype == np.float64:
        assert math.isnan(fx[1](np.array([1.0] * (at % 150) + [bad])))


def test_zeros_of_either_sign(fx):
    assert fx[0](np.array([0.0, -0.0, 0.0])) == 0.0
    assert fx[0](np.array([-0.0] * 64, np.float32)) == 0.0


def test_no_further_off_than_a_tree_of_fp64_additions(fx):
    """Over random summands of mixed signs and magnitudes the worst error, relative to the sum of
    magnitudes, is below that of a pairwise FP64 sum."""
    rng = np.random.default_rng(9)
    worst = [0.0, 0.0]
    for _ in range(200):
        a = rng.standard_normal(1024) * 2.0 ** rng.uniform(-20, 0, 1024)
        exact, mag, t = math.fsum(a), math.fsum(np.abs(a)), a
        while t.size > 1:
            t = t[: t.size // 2] + t[t.size // 2:]
        for k, s in enumerate((fx[0](a), t[0])):
            worst[k] = max(worst[k], abs(s - exact) / mag)
    assert worst[0] <= worst[1]
    assert worst[0] <= 2.0 ** -53
