"""CPU checks of the fixed-point PxPyPzE pair mass (csrc/cart_fixed.cuh), compiled for the host from the
same source, where its limbs change hands: components from none to 90 binades below the largest (20
is the last that one shift per limb places), exact zeros and denormals next to normal values, every
combination of signs.  Tolerance: 2^-44 relative to the binary128 mass in FP64 and one rounding in
FP32, the bounds the fast path states."""
import numpy as np
import pytest

import gvx_synth as syn
from test_ff_host import _cart_fixed, ffh  # noqa: F401 (fixture)


def _legs(which, n):
    g = syn.rng(541)
    a, b = syn.pxpypze(g, n), syn.pxpypze(g, n)
    if which == "zeros":
        a[:, 0] = b[::2, 1] = a[1::2, 2] = 0.0
    elif which == "denormals":
        a[:, 0], b[::2, 1], b[1::2, 2] = 5e-324, -1e-310, -0.0
    elif which == "signs":
        b[:, :3] *= np.where(g.random((n, 3)) < 0.5, -1.0, 1.0)
        a[::3, 3] *= -1.0
    else:
        k = int(which)
        b *= 2.0 ** -k
        a[::2, 1] *= 2.0 ** -k
    return np.ascontiguousarray(a), np.ascontiguousarray(b)


@pytest.mark.parametrize("which", ["1", "12", "19", "20", "21", "22", "30", "31", "33", "52", "60", "83",
                                   "84", "90", "zeros", "denormals", "signs"])
def test_pxpypze_mass_against_oracle(ffh, orc, which):  # noqa: F811
    a, b = _legs(which, 20000)
    for x, y in ((a, b), (b, a)):
        m, ok, m32, ok32 = _cart_fixed(ffh, x, y)
        ref = orc.mass_cart_def(x, y, "pxpypze")
        assert np.max(np.abs(m - ref)[ok] / np.abs(ref[ok])) <= 2.0 ** -44
        x32, y32 = syn.to_f32(x).astype(np.float64), syn.to_f32(y).astype(np.float64)
        ref32 = orc.mass_cart_def(x32, y32, "pxpypze")
        big = ok32 & (np.abs(ref32) > 1e-30)
        assert np.max(np.abs(m32.astype(np.float64) - ref32)[big] / np.abs(ref32[big])) <= 2.0 ** -24 * 1.01
        assert np.array_equal(m, _cart_fixed(ffh, y, x)[0], equal_nan=True)  # symmetric, bit for bit
