"""The FP64 force kernel's reciprocal square root (csrc/nb_rsqrt.cuh) by itself, against
exact integer arithmetic: the header is compiled into a small program of its own with the
force kernel's flags. Bounds: in [2^-120, 2^120) half an ulp for the last rounding, 2^-63.4
relative for the step's truncation (below 2^-10.4 ulp) and 2^-73 for its other roundings,
0.501 ulp; outside, CUDA's 1 ulp for rsqrt(). A step without its third-order term is far
outside that bound."""
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import ics

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _ulps(q, r2):
    """|q - r2^(-1/2)| in ulps of q, from q^2 r2 - 1 in integers (the square of the error is nothing)."""
    (a, b), (c, d) = float(q).as_integer_ratio(), float(r2).as_integer_ratio()
    num, den = a * a * c, b * b * d
    return abs((num - den) / (2 * den)) * float(q) / math.ulp(q)


def _mantissas(rng, count):
    edge = [1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -23, 2.0 - 2.0 ** -23, 1.5, 1.0 + 2.0 ** -24 - 2.0 ** -52]
    return np.concatenate([edge, 1.0 + rng.uniform(count)])


@pytest.fixture(scope="module")
def rsqrt(tmp_path_factory):
    import paper_0711_0643_gb300._build as B
    d = tmp_path_factory.mktemp("rsqrt")
    exe, fin, fout = (str(d / s) for s in ("check", "in", "out"))
    flags = dict(B.SOURCES)["nb_force.cu"]
    subprocess.run([B.nvcc(), *B.ARCH, *B.COMMON, *flags, "-I", B.CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "rsqrt_f64_check.cu")], check=True)

    def call(x):
        np.asarray(x, dtype=np.float64).tofile(fin)
        subprocess.run([exe, fin, fout], check=True)
        return np.fromfile(fout)
    return call


@pytest.mark.gpu
def test_inside_the_fp32_range(rsqrt):
    rng = ics.SplitMix64(61)
    x = np.concatenate([np.ldexp(_mantissas(rng, 400), e) for e in range(-120, 120)])
    assert max(_ulps(q, r) for q, r in zip(rsqrt(x), x)) <= 0.501


@pytest.mark.gpu
def test_outside_it(rsqrt):
    rng = ics.SplitMix64(62)
    lo = np.concatenate([np.ldexp(_mantissas(rng, 20), e) for e in range(-1074, -120)])
    hi = np.concatenate([np.ldexp(_mantissas(rng, 20), e) for e in range(120, 1024)])
    x = np.concatenate([lo[lo > 0], hi, [5e-324, np.finfo(float).max]])
    assert max(_ulps(q, r) for q, r in zip(rsqrt(x), x)) <= 1.0
    got = rsqrt([0.0, np.inf, np.nan, -1.0, -2.0 ** -130, -np.inf])
    assert got[0] == np.inf and got[1] == 0.0 and np.isnan(got[2:]).all()


def test_the_bound_sees_the_third_order_term():
    """The same step in exact arithmetic on the CPU, rounded once, with and without 3/8 e^2."""
    rng = ics.SplitMix64(63)
    for r2 in _mantissas(rng, 200):
        q0 = Fraction(float(np.float32(1.0 / math.sqrt(r2)) * np.float32(1.0 + 2.0 ** -22)))   # 2 ulp off
        e = 1 - Fraction(float(r2)) * q0 * q0
        assert _ulps(float(q0 + q0 * e * (Fraction(1, 2) + Fraction(3, 8) * e)), r2) <= 0.501
        assert _ulps(float(q0 + q0 * e / 2), r2) > 100.0
