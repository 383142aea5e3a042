"""CPU checks of the fixed-point PxPyPzE pair mass (csrc/cart_fixed.cuh) at both ends of the scale
exponents it takes (+-100 for FP32 legs, +-900 for FP64 ones), with exact zeros among the components:
a zero is zero at every scale, however few binades lie between the largest component and the format's
exponent field of 0.  Tolerance: 2^-44 relative to the binary128 mass in FP64 and one rounding in
FP32, the bounds the fast path states."""
import numpy as np
import pytest

import gvx_synth as syn
from test_ff_host import _cart_fixed, ffh  # noqa: F401 (fixture)


def _legs(s, dtype, n):
    """Pairs whose largest component lies in [2^s, 2^(s+1)), light and heavy, a third of the components
    zero and the others normal."""
    g = syn.rng(551)
    a, b = syn.pxpypze(g, n), syn.pxpypze(g, n)
    top = np.exp2(np.floor(np.log2(np.max(np.abs(np.hstack([a, b])), axis=1))))[:, None]
    a, b = np.ldexp(a / top, s), np.ldexp(b / top, s)
    a, b = (np.where(g.random((n, 4)) < 0.33, g.choice([0.0, -0.0], (n, 4)), v) for v in (a, b))
    b[::4] = 0.0  # a leg at rest, up to 25 binades below the scale
    b[::4, 3] = np.ldexp(1.0, s - g.integers(0, 26, len(b[::4])))
    a[::8] = 0.0  # with a massless one
    a[::8, 0] = a[::8, 3] = np.ldexp(1.5, s)
    a, b = (v.astype(dtype).astype(np.float64) for v in (a, b))
    return tuple(np.where(np.abs(v) < np.finfo(dtype).tiny, 0.0, v) for v in (a, b))


def _check(got, ok, ref, tol, least=0.5):
    hit = ok & (ref != 0.0)
    assert hit.mean() > least
    assert np.max(np.abs(got - ref)[hit] / np.abs(ref[hit])) <= tol


@pytest.mark.parametrize("s", [-100, -99, -98, -97, -60, 0, 99, 100])
def test_f32_scales(ffh, orc, s):  # noqa: F811
    a, b = _legs(s, np.float32, 8000)
    for x, y in ((a, b), (b, a)):
        _, _, m, ok = _cart_fixed(ffh, x, y)
        _check(m.astype(np.float64), ok, orc.mass_cart_def(x, y, "pxpypze"), 2.0 ** -24 * 1.01)


@pytest.mark.parametrize("s", [-900, -899, 0, 899, 900])
def test_f64_scales(ffh, orc, s):  # noqa: F811
    a, b = _legs(s, np.float64, 8000)
    for x, y in ((a, b), (b, a)):
        m, ok, _, _ = _cart_fixed(ffh, x, y)
        _check(m, ok, orc.mass_cart_def(x, y, "pxpypze"), 2.0 ** -44)


@pytest.mark.parametrize("s", [-100, -97, -80, -60, -44, -43, -42])
def test_f32_denormal_components(ffh, orc, s):  # noqa: F811
    """A denormal component counts like any other: a pair with one is right, or declined where it would
    lie above the units (2^-83 of the scale)."""
    g = syn.rng(553)
    a, b = _legs(s, np.float32, 8000)
    for v in (a, b):
        low = g.random(v.shape) < 0.15
        low[:, 3] = False
        v[low] = (g.integers(1, 1 << 23, low.sum()) * g.choice([-1.0, 1.0], low.sum())) * 2.0 ** -149
    _, _, m, ok = _cart_fixed(ffh, a, b)
    _check(m.astype(np.float64), ok, orc.mass_cart_def(a, b, "pxpypze"), 2.0 ** -24 * 1.01, 0.2)
