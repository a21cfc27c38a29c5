"""The reduced-range integer-pipe functions as the kernels run them: the device
build of emu::*_mid, with the MUFU pipe's starts, on the operands of the host
test.  Products and sums have the bits of the DMUL / DADD instructions; the
reciprocal lies within 1/2 + 2^-4 units in the last place, ab/(a+b) and the root
within 1/2 + 2^-3; the flags are those of the host build."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest
import torch

from test_emu64_mid_host import _mid, _pairs, _ulps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe():
    from paper_1512_03662_gb300 import build
    build.build()
    L = ctypes.CDLL(build.PROBE_LIB)
    L.fp64_mid_check.restype = ctypes.c_int
    L.fp64_mid_check.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_longlong, ctypes.c_void_p]
    return L


@pytest.mark.parametrize("seed", [1, 5])
def test_the_functions_that_the_kernels_call(probe, seed):
    a, b = _pairs(seed)
    # dense starts of the reciprocal and the root: every leading part of the significand
    lead = 1.0 + np.arange(1 << 14) / (1 << 14)
    a, b = np.concatenate([a, lead, 4 * lead - 2.0 ** -40]), np.concatenate([b, lead[::-1], lead])
    n = len(a)
    ag, bg = torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda")
    out = torch.empty(5, n, dtype=torch.float64, device="cuda")
    okg = torch.empty(n, dtype=torch.uint8, device="cuda")
    assert probe.fp64_mid_check(*(ctypes.c_void_p(t.data_ptr()) for t in (ag, bg, out, okg)), n, None) == 0
    prod, total = (ag * bg).cpu().numpy(), (ag + bg).cpu().numpy()
    torch.cuda.synchronize()
    m, r, h, q, p = out.cpu().numpy()
    ok = okg.cpu().numpy()
    za, zb = a == 0, b == 0
    pair = (_mid(a) | za) & (_mid(b) | zb)
    for bit, want in ((1, pair), (2, _mid(a)), (4, pair), (8, _mid(a) & (a > 0)), (16, pair)):
        assert np.array_equal((ok & bit) != 0, want), bit
    assert (m.view(np.int64) == prod.view(np.int64))[pair].all()
    assert ((p.view(np.int64) == total.view(np.int64)) | ((p == 0) & (total == 0)))[pair].all()
    worst = max(_ulps(r[i], 1 / Fraction(float(a[i]))) for i in np.flatnonzero(_mid(a)))
    assert worst <= Fraction(1, 2) + Fraction(1, 16), float(worst)
    same = pair & ~za & ~zb & (np.signbit(a) == np.signbit(b))
    assert (h[pair & ~same] == 0).all()
    exact = lambda x, y: x * y / (x + y)  # noqa: E731
    worst = max(_ulps(h[i], exact(Fraction(float(a[i])), Fraction(float(b[i])))) for i in np.flatnonzero(same))
    assert worst <= Fraction(1, 2) + Fraction(1, 8), float(worst)
    t = Fraction(1, 2) + Fraction(1, 8)
    for i in np.flatnonzero(_mid(a) & (a > 0)):
        y, u = Fraction(float(q[i])), Fraction(float(np.spacing(q[i])))
        assert (y - t * u) ** 2 <= Fraction(float(a[i])) <= (y + t * u) ** 2, (a[i], q[i])
