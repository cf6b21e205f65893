"""The division-free scalar helpers of the recurrences and of the inner part (square
root and inverse from one reciprocal square root; beta, gamma and their inverses of a
complex delta; inverses of pivots) over the whole exponent range: subnormals, both ends,
zero real or imaginary part.

Bounds, with u = 2^-53 and relative in the complex modulus, from the operations of each
helper: rsqrt is good to 1 ulp (2u), the Newton correction to half an ulp and the
squared error (2u, twice that where the residual of a subnormal is rounded); csqrt_scalars
chains two reciprocal square roots and at most one complex product (12u); an inverse of a
real pivot 1 ulp (2u), or the correctly rounded quotient; of a complex one the norm (2u),
its inverse (2u) and a product (u) (6u; Smith's quotient at the ends of the range 16u).
"""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_0912_4457_gb300 import build  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53
LD, CLD = np.longdouble, np.clongdouble


@pytest.fixture(scope="module")
def values(tmp_path_factory):
    """(z, out): the inputs and the helpers' 18 results of each"""
    exe = str(tmp_path_factory.mktemp("scalars") / "scalar_harness")
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O3", "-I", build.CSRC, "-I", build.INCLUDE,
                    os.path.join(ROOT, "tests", "cpp", "scalar_harness.cu"), "-o", exe], check=True)
    rng = np.random.default_rng(5)
    m = 4000
    ex = rng.integers(-1070, 1022, m)
    x = np.ldexp(rng.uniform(1, 2, m) * rng.choice([-1, 1], m), ex)
    y = np.ldexp(rng.uniform(1, 2, m) * rng.choice([-1, 1], m), np.clip(ex + rng.integers(-60, 60, m), -1074, 1022))
    one = np.ldexp(rng.uniform(1, 2, 500), rng.integers(-3, 4, 500))
    ends = np.array([2.0 ** e for e in (-1074, -1060, -1023, -1022, -1021, -1012, -1002, -1001, -1000, -999, -1, 0, 1, 999,
                                        1000, 1001, 1002, 1021, 1022)] + [np.finfo(float).max / 2])
    z = np.concatenate([x + 1j * y, one * np.exp(1j * rng.uniform(-np.pi, np.pi, 500)), ends + 0j, -ends + 0j, 1j * ends,
                        -1j * ends, ends * (1 + 1j), ends * (-1 + 1e-9j)])
    text = "%d\n" % len(z) + "".join("%.17g %.17g\n" % (v.real, v.imag) for v in z)
    res = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    out = np.array([float(t) for t in res.split()]).reshape(len(z), 18)
    return z, out


def err(got, ref):
    """relative, beyond half a unit of the smallest subnormal; infinite where the reference is"""
    with np.errstate(all="ignore"):
        d = np.abs(np.asarray(got, CLD) - ref) - LD(2.0) ** -1074
        return np.where(np.abs(ref) > np.finfo(float).max, np.where(np.isfinite(got), np.inf, 0), np.maximum(d, 0) / np.abs(ref))


def cpx(o, c):
    got = np.empty(len(o), CLD)
    got.real, got.imag = o[:, c], o[:, c + 1]
    return got


def test_square_root_and_inverse(values):
    z, o = values
    x = np.abs(z.real)
    keep = x > 0
    x, s, inv = x[keep], o[keep, 0], o[keep, 1]
    r = np.sqrt(np.asarray(x, LD))
    tiny = x < 2.0 ** -960
    assert err(s, r)[~tiny].max() <= 2 * U and err(s, r)[tiny].max() <= 4 * U
    assert err(inv, 1 / r).max() <= 2 * U


def test_hermitian_step_scalars(values):
    z, o = values
    pos = z.real > 0
    np.testing.assert_array_equal(o[pos, 16], o[pos, 0])
    np.testing.assert_array_equal(o[pos, 17], o[pos, 1])
    assert (o[~pos, 17] == -1.0).all()   # no positive delta: breakdown


def test_two_sided_scalars(values):
    z, o = values
    d = np.asarray(z, CLD)
    scale = np.exp2(np.floor(np.log2(np.maximum(np.abs(z.real), np.abs(z.imag)).astype(LD)) / 2) * 2).astype(LD)
    beta = np.sqrt(d / scale) * np.sqrt(scale)
    beta = np.where((z.imag == 0) & (z.real < 0), np.abs(beta) * CLD(1j), beta)   # the cut belongs to Im >= 0
    gamma = np.conj(d) / beta
    for c, ref in ((2, beta), (4, gamma), (6, 1 / beta), (8, 1 / gamma)):
        assert err(cpx(o, c), ref).max() <= 12 * U, c


def test_real_pivots(values):
    z, o = values
    x = z.real
    keep = x != 0
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(o[keep, 11], 1.0 / x[keep])
    assert err(o[keep, 10], 1 / np.asarray(x[keep], LD)).max() <= 2 * U


def test_complex_pivots(values):
    z, o = values
    big = np.maximum(np.abs(z.real), np.abs(z.imag))
    mid = (big >= 2.0 ** -1000) & (big < 2.0 ** 1001)
    s = np.asarray(big, LD)
    w = np.asarray(z, CLD) / s
    ref = np.conj(w) / (w.real * w.real + w.imag * w.imag) / s
    inside = np.abs(ref) < LD(2.0) ** 1020
    for c in (12, 14):
        e = err(cpx(o, c), ref)
        assert e[mid].max() <= 6 * U, c
        assert e[~mid & inside].max() <= 16 * U, c
