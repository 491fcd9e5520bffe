"""The FP64 reciprocal and reciprocal square root (rb_fp64.cuh) against the
exact values over the whole exponent range, both sides of the exponents where
they change over to the library's functions, and through the FP64 walk at
distances whose squares leave the normal range."""
import ctypes
import os
import subprocess
from fractions import Fraction
from math import isqrt

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1110_4876_gb300 import build

    out = str(tmp_path_factory.mktemp("fp64") / "fp64_probe.so")
    # contraction off, as in the walks' translation units
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-fmad=false", "-I", build.CSRC, "-shared", "-Xcompiler",
                    "-fPIC", "-o", out, os.path.join(HERE, "fp64_probe.cu")], check=True)
    f = ctypes.CDLL(out).fp64_probe

    def run(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        a, b = np.empty_like(x), np.empty_like(x)
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, a, b)]
        assert f(p[0], ctypes.c_int(len(x)), p[1], p[2]) == 0
        return a, b

    return run


def _numbers():
    g = np.random.default_rng(7)
    sig = g.integers(0, 1 << 52, 40_000, dtype=np.uint64)
    exp = g.integers(1, 2047, 40_000, dtype=np.uint64)
    edge = np.repeat(np.array([1, 2, 63, 64, 65, 1022, 1023, 1024, 1981, 1982, 1983, 2045, 2046], np.uint64), 40)
    esig = g.integers(0, 1 << 52, len(edge), dtype=np.uint64)
    esig[::40] = 0
    esig[1::40] = (1 << 52) - 1
    sub = np.concatenate([g.integers(1, 1 << 52, 40, dtype=np.uint64), np.array([1, (1 << 52) - 1], np.uint64)])
    bits = np.concatenate([exp << np.uint64(52) | sig, edge << np.uint64(52) | esig, sub])
    return bits.view(np.float64)


def _ulps(y, v):
    """|y - v| in units of the last place of y."""
    return abs(Fraction(y) - v) / Fraction(float(np.spacing(y)))


def _rsqrt(f):
    """1/sqrt(f) to 2^-127 relative."""
    k = max(0, 128 + (f.numerator.bit_length() - f.denominator.bit_length()) // 2)
    return Fraction(isqrt((f.denominator << (2 * k)) // f.numerator), 1 << k)


def test_reciprocals_to_the_last_place(probe):
    """Worst errors in units of the last place, for estimates good to 2^-18 or
    better.  1/x: h is one rounding of a number below 2^-18, the series leaves
    h^3 < 2^-54 (0.5 units at most), the last operation rounds once (0.5): at
    most 1.  1/sqrt(x): x y is rounded (2^-53 in h, 2^-54 in the result, 0.5
    units at most), the series leaves 5/16 h^3 with h < 2^-17 (2^-52.7, below
    0.7), the last operation rounds once: at most 2."""
    x = _numbers()
    rcp, rsq = probe(x)
    worst = [Fraction(0), Fraction(0)]
    for v, a, b in zip(map(Fraction, x.tolist()), rcp.tolist(), rsq.tolist()):
        if np.isfinite(a):
            worst[0] = max(worst[0], _ulps(a, 1 / v))
        else:
            assert 1 / v > Fraction(float(np.finfo(np.float64).max))
        worst[1] = max(worst[1], _ulps(b, _rsqrt(v)))
    print("worst units: 1/x", float(worst[0]), "1/sqrt(x)", float(worst[1]))
    assert worst[0] <= 1
    assert worst[1] <= 2


def test_reciprocals_of_special_values(probe):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -2.5, -1e-310])
    rcp, rsq = probe(x)
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(rcp, 1.0 / x)
    np.testing.assert_array_equal(rsq, [np.inf, -np.inf, 0.0, np.nan, np.nan, np.nan, np.nan])


@pytest.mark.parametrize("d", [1e160, 1e-156])
def test_fp64_walk_beyond_the_range_of_squares(d):
    """Two bodies so far apart that r^2 is infinite exert no force, and so near
    that it is subnormal still have their potential, -1/d to the few bits that
    r^2 keeps (2^-40 at 1e-312)."""
    from paper_1110_4876_gb300 import build, rb

    build.build()
    x, zero, one = np.array([-0.5 * d, 0.5 * d]), np.zeros(2), np.ones(2)
    sim = rb.Sim(G=1.0, box=(4 * d,) * 3, theta=0.5, gravity=1, walk=rb.RB_WALK_FP64)
    sim.set_particles((x, zero, zero, zero, zero, zero, one, zero))
    if d > 1.0:
        assert np.array_equal(sim.gravity(), np.zeros((2, 3)))
    W = sim.energy_terms()[2]
    assert W == pytest.approx(-1.0 / d if d < 1.0 else 0.0, rel=2.0 ** -36)
