"""CPU checks of the float-float PxPyPzM pair mass (csrc/cart_pxpypzm.cuh), compiled for the host from
the same source, against the binary128 oracle where its projection of one leg on the other can go
wrong: angles from 1 down to 1e-10 (the projection is good to about 2^-22), legs near rest, opposite
legs, legs along an axis (exact zeros), scales up to 60 binades apart, massless legs.

Tolerance: 2^-43 relative in FP64 and one rounding in FP32, the bounds the fast path states."""
import numpy as np
import pytest

import gvx_synth as syn
from test_ff_host import _cart_fixed, ffh  # noqa: F401 (fixture)

CASES = ["angle1", "angle1e-3", "angle2e-7", "angle1e-10", "rest", "opposite", "axis", "gap", "massless"]


def _legs(which, n):
    g = syn.rng(521)
    a, b = syn.pxpypze(g, n), syn.pxpypze(g, n)
    a[:, 3], b[:, 3] = g.uniform(0, 10, n), g.uniform(0, 10, n)
    if which.startswith("angle"):
        t = float(which[5:])
        b[:, :3] = a[:, :3] * g.uniform(0.5, 2.0, (n, 1)) * (1 + t * g.uniform(-1, 1, (n, 3)))
    elif which == "rest":
        a[:, :3] *= 2.0 ** g.uniform(-80, -10, (n, 1))
    elif which == "opposite":
        b[:, :3] = -a[:, :3] * g.uniform(0.5, 2.0, (n, 1))
    elif which == "axis":
        a[:, :2] = 0.0
        b[::2, 1:3] = 0.0
        b[1::2, 2] = 0.0
    elif which == "gap":
        b *= 2.0 ** g.integers(-40, 40, (n, 1))
    else:
        a[:, 3] = 0.0
        b[::2, 3] = 0.0
    return np.ascontiguousarray(a), np.ascontiguousarray(b)


@pytest.mark.parametrize("which", CASES)
def test_pxpypzm_mass_against_oracle(ffh, orc, which):  # noqa: F811
    for a, b in (_legs(which, 20000), _legs(which, 20000)[::-1]):
        m, ok, _, _ = _cart_fixed(ffh, a, b, coords=1)
        ref = orc.mass_cart_def(a, b, "pxpypzm")
        assert ok.mean() > 0.99
        assert np.max(np.abs(m - ref)[ok] / ref[ok]) <= 2.0 ** -43
        a32, b32 = syn.to_f32(a).astype(np.float64), syn.to_f32(b).astype(np.float64)
        _, _, m32, ok32 = _cart_fixed(ffh, a32, b32, coords=1)
        ref32 = orc.mass_cart_def(a32, b32, "pxpypzm")
        big = ok32 & (ref32 > 1e-30)
        assert np.max(np.abs(m32.astype(np.float64) - ref32)[big] / ref32[big]) <= 2.0 ** -24 * 1.01
