"""The kernels' own arithmetic, function by function, against exact values:
the functions of the device headers compiled into a small library of their own
(arith_probe.cu)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2511_06152_gb300 import build as b
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "arith_probe.cu")
    so = str(tmp_path_factory.mktemp("probe") / "libarith_probe.so")
    subprocess.run([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    "-I" + b.CSRC, "-I" + os.path.join(b.ROOT, "include"), "-shared", "-o", so, src], check=True)
    return ctypes.CDLL(so)


def _call(f, inp, out, *n):
    inp = np.ascontiguousarray(inp)
    assert f(ctypes.c_void_p(inp.ctypes.data), ctypes.c_void_p(out.ctypes.data), *n) == 0
    return out


def test_binary64_reciprocal_is_the_quotient(probe):
    """1 / z of the cost and the linearisation, from just above the smallest
    depth (1e-6) on: the correctly rounded quotient, 0 for an infinite depth."""
    rng = np.random.Generator(np.random.PCG64(1))
    x = np.concatenate([np.nextafter(1e-6, 1.0) * (1 + rng.random(100_000)), 300.0 * (0.5 + rng.random(300_000)),
                        np.ldexp(1 + rng.random(400_000), rng.integers(-20, 1023, 400_000)),
                        2.0 - 2.0 ** -np.arange(1.0, 53.0), [np.inf]])
    assert np.array_equal(_call(probe.probe_recip, x, np.empty_like(x), len(x)), 1.0 / x)


def test_difference_of_double_floats_rounds_once(probe):
    """X - T of a point and an image centre in grid coordinates (5e5, 5e6 m),
    1e-3 .. 1e3 m apart: rounded to binary32 from the exact difference.  The
    accurate sum's relative error of 3 2^-48 is 3 2^-24 ulp of the result."""
    rng = np.random.Generator(np.random.PCG64(2))
    n = 1_000_000
    X = np.where(rng.random(n) < 0.5, 5e5, 5e6) * (1 + 0.1 * rng.random(n))
    T = X + 10.0 ** rng.uniform(-3, 3, n) * rng.choice([-1, 1], n)
    ab = np.empty((n, 4), np.float32)
    for i, v in ((0, X), (2, -T)):
        ab[:, i] = v
        ab[:, i + 1] = v - ab[:, i].astype(np.float64)
    got = _call(probe.probe_sum, ab, np.empty(n, np.float32), n).astype(np.float64)
    w = ab.astype(np.float64)  # both partial sums, and the total, are exact in binary64
    exact = (w[:, 0] + w[:, 2]) + (w[:, 1] + w[:, 3])
    ulp = np.spacing(np.abs(exact).astype(np.float32)).astype(np.float64)
    assert (np.abs(got - exact) <= (0.5 + 2.0 ** -20) * ulp).all()


@pytest.mark.parametrize("exponent", [-96, -37, 0, 1, 2])
def test_pivot_reciprocal_is_as_accurate_as_the_quotients(probe, exponent):
    """1 / d of a pivot (double-float, Newton's iteration from the hardware's
    approximation) over every binary32 significand: no further off than the
    reciprocal that starts from the correctly rounded quotient."""
    fast, ref = _call(probe.probe_df_recip, np.array([2.0 ** exponent], np.float32), np.empty(2))
    assert 0 < ref < 2.0 ** -45  # e^2, |e| <= 2^-23 (half an ulp of r, half an ulp of the high word), and its roundings
    assert fast <= ref, (np.log2(fast), np.log2(ref))


def test_observations_of_no_weight_add_nothing(probe):
    """Behind the image, or so far off that the squared error overflows: the
    contribution to the point's step is zero."""
    x = np.array([10.0, 1e3, 1e5, 4e6], np.float32)
    behind = np.zeros((4, 11), np.float32)
    behind[:, 0], behind[:, 1], behind[:, 2] = x, 0.3 * x, -0.2 * x
    front = np.zeros((3, 11), np.float32)  # 100 m to the side, 1 mm .. 0.1 mm in front
    front[:, 0], front[:, 2] = 100.0, (1e-3, 3e-4, 1e-4)
    rows = np.concatenate([behind, front])
    rows[:, 5:] = (1e-4, -2e-4, 3e-4, 0.01, 0.02, -0.03)
    g = _call(probe.probe_obs_step, rows, np.empty((7, 3), np.float32), 7)
    assert (g == 0).all(), g
