"""The reduced-range products, the reciprocal, the limited slope and the root on the
integer pipes (emu64.cuh), built for the host with g++, against exact integer
and rational arithmetic: products bit for bit with the IEEE ones, the
reciprocal within 1/2 + 2^-4 units in the last place and ab/(a+b) within
1/2 + 2^-3, the root too (the bounds that their fixed-point errors of at most
2^-58 and 2^-56 leave), for every start that the 24-bit approximation may give (a unit
off), and never a value outside the range taken without a cleared flag."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from emu_cases import emu_operands

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1512_03662_gb300", "csrc")


@pytest.fixture(scope="module", params=[0, 1, -1])
def emu(request, tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("emu") / "libemu64mid.so")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    f"-DEMU_RCP_ERROR={request.param}", os.path.join(HERE, "emu64_mid_host.cpp"), "-o", out],
                   check=True)
    L = ctypes.CDLL(out)
    L.emu64_mid_host.restype = None
    L.emu64_mid_host.argtypes = [ctypes.c_void_p] * 8 + [ctypes.c_longlong]
    return L


def _run(L, a, b):
    n = len(a)
    m, r, h, q, p = (np.empty(n) for _ in range(5))
    ok = np.empty(n, dtype=np.uint8)
    L.emu64_mid_host(*(x.ctypes.data for x in (a, b, m, r, h, q, p, ok)), n)
    return m, r, h, q, p, ok


def _mid(x):
    return (np.abs(x) >= 2.0 ** -500) & (np.abs(x) < 2.0 ** 500)


def _ulps(got, exact):
    """|got - exact| in units in the last place of got (exact: Fraction)."""
    return abs(Fraction(float(got)) - exact) / Fraction(float(np.spacing(abs(got))))


def _pairs(seed):
    """Operands of the listed classes plus same-sign pairs over every exponent
    gap, equal operands, powers of two and all-ones significands."""
    a, b = emu_operands(1 << 14, seed)
    rng = np.random.default_rng(seed + 100)
    k = 1 << 13
    x = np.ldexp(rng.uniform(1, 2, k), rng.integers(-60, 60, k)) * rng.choice([-1.0, 1.0], k)
    gap = rng.integers(-70, 70, k)
    y = np.ldexp(np.abs(x), gap) * rng.uniform(0.5, 1, k) * np.sign(x)
    one = 2.0 - 2.0 ** -52
    edge = np.array([1.0, one, 1.0 + 2.0 ** -52, 1.5, 2.0 ** -499, 2.0 ** 499, one * 2.0 ** 499, 1.0 - 2.0 ** -53])
    e0, e1 = np.meshgrid(edge, edge)
    return (np.concatenate([a, x, x, e0.ravel(), -e0.ravel()]),
            np.concatenate([b, y, x, e1.ravel(), -e1.ravel()]))


@pytest.mark.parametrize("seed", [1, 2])
def test_products_reciprocals_and_slopes(emu, seed):
    a, b = _pairs(seed)
    m, r, h, q, p, ok = _run(emu, a, b)
    za, zb = a == 0, b == 0
    with np.errstate(all="ignore"):
        ref = a * b
    # the flags: exactly the moderate operands and zeros
    assert np.array_equal((ok & 1) != 0, (_mid(a) | za) & (_mid(b) | zb))
    assert np.array_equal((ok & 2) != 0, _mid(a))
    assert np.array_equal((ok & 4) != 0, (_mid(a) | za) & (_mid(b) | zb))
    good = (ok & 1) != 0
    assert (m.view(np.int64) == ref.view(np.int64))[good].all()
    pick = np.flatnonzero((ok & 2) != 0)
    worst = max(_ulps(r[i], 1 / Fraction(float(a[i]))) for i in pick)
    assert worst <= Fraction(1, 2) + Fraction(1, 16), float(worst)
    same = ((ok & 4) != 0) & ~za & ~zb & (np.signbit(a) == np.signbit(b))
    assert (h[((ok & 4) != 0) & ~same] == 0).all()
    worst = 0
    for i in np.flatnonzero(same):
        x, y = Fraction(float(a[i])), Fraction(float(b[i]))
        worst = max(worst, _ulps(h[i], x * y / (x + y)))
    assert worst <= Fraction(1, 2) + Fraction(1, 8), float(worst)
    # sqrt: q is within t units u of the root when (q - t u)^2 <= a <= (q + t u)^2
    assert np.array_equal((ok & 8) != 0, _mid(a) & (a > 0))
    t = Fraction(1, 2) + Fraction(1, 8)
    for i in np.flatnonzero(ok & 8):
        y, u = Fraction(float(q[i])), Fraction(float(np.spacing(q[i])))
        assert (y - t * u) ** 2 <= Fraction(float(a[i])) <= (y + t * u) ** 2, (a[i], q[i])
    # sums: the IEEE one or, where bits fell below the frame, within 1/2 + 2^-9
    assert np.array_equal((ok & 16) != 0, (_mid(a) | za) & (_mid(b) | zb))
    with np.errstate(all="ignore"):
        ref = a + b
    for i in np.flatnonzero(((ok & 16) != 0) & (p.view(np.int64) != ref.view(np.int64))):
        x = Fraction(float(a[i])) + Fraction(float(b[i]))
        if x == 0:
            assert p[i] == 0
        else:
            assert _ulps(p[i], x) <= Fraction(1, 2) + Fraction(1, 512), (a[i], b[i], p[i])


@pytest.mark.parametrize("seed", [3, 4])
def test_sums_are_correctly_rounded(emu, seed):
    """add_mid gives the bits of the IEEE sum (up to the sign of a zero) for every
    exponent gap, ties whose lower operand lies below the 64-bit frame
    included: half a unit in the last place of the larger operand, exactly, and
    with one more bit far below."""
    a, b = _pairs(seed)
    rng = np.random.default_rng(seed)
    k = 1 << 14
    x = np.ldexp(rng.uniform(1, 2, k), rng.integers(-40, 40, k))
    half = np.spacing(x) / 2
    far = half * (1 + np.ldexp(1.0, -rng.integers(1, 53, k)))
    near = half * (1 - np.ldexp(1.0, -rng.integers(1, 54, k)))
    s = rng.choice([-1.0, 1.0], 6 * k)
    a = np.concatenate([a, x, x, x, half, far, near])
    b = np.concatenate([b, half, far, near, x, x, x])
    b[-6 * k:] *= s
    p, ok = (lambda r: (r[4], r[5]))(_run(emu, a, b))
    with np.errstate(all="ignore"):
        ref = a + b
    good = (ok & 16) != 0
    assert good[-6 * k:].all()
    assert ((p == ref) & ((p.view(np.int64) == ref.view(np.int64)) | (ref == 0)))[good].all()
