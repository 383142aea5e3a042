"""CPU checks of the jagged adjoint's pair terms (csrc/event_lc_grad.cuh) where an angle difference is small:
d/dphi is proportional to sin(d_phi) and has to be right by itself however small it is beside d_eta, and so
has d/deta of two legs alike but for the sign of eta, whose only term is sinh(d_eta).  Tolerance: 1e-12
relative per component, the adjoint's gate."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def enh(tmp_path_factory):
    from paper_2312_02756_gb300 import gen_tables
    out = str(tmp_path_factory.mktemp("enh"))
    gen_tables.write(os.path.join(out, "gvx_tables.inc"))
    lib = os.path.join(out, "enh.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + out,
                    os.path.join(HERE, "event_near_harness.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _grads(lib, name, a, b, gm):
    """(grad a, grad b, ok, FP64 differences taken) of the harness function `name`."""
    n = len(a)
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    ga, gb, ok, asked = np.empty_like(a), np.empty_like(a), np.empty(n, np.uint8), np.zeros(n, np.uint8)
    args = [p(a), p(b), p(gm), ctypes.c_int64(n), p(ga), p(gb), p(ok)]
    getattr(lib, name)(*args, *([p(asked)] if name == "enh_pairs" else []))
    return ga, gb, ok.astype(bool), asked.astype(bool)


def near_pairs(angle, size, n=20_000):
    """Pairs whose phi (angle 2) or eta (angle 1) are 1e-2 to 1e-18 apart around 0 (size "small") or
    around values from 2^-8 to 3 (size "large"), and whose other angles are 0.1 to 2 apart."""
    g = syn.rng(571)
    a, b = syn.ptetaphim(g, n), syn.ptetaphim(g, n)
    d = 10.0 ** g.uniform(-18, -2, n) * g.choice([-1.0, 1.0], n)
    other = 3 - angle
    b[:, other] = np.clip(a[:, other], -1, 1) + g.uniform(0.1, 2.0, n)
    a[:, other] = np.clip(a[:, other], -1, 1)
    f = g.uniform(0, 1, n)
    if size == "small":
        a[:, angle], b[:, angle] = f * d, (f - 1) * d
        a[::5, angle] = 0.0
    else:
        base = np.exp2(g.uniform(-8, 1.5, n)) * g.choice([-1.0, 1.0], n)
        a[:, angle], b[:, angle] = base, base + d
    if angle == 1:  # W = 0: the same pt and m, and |eta| the same
        b[:, [0, 3]] = a[:, [0, 3]]
        if size == "small":
            a[:, 1], b[:, 1] = 0.5 * d, -0.5 * d
    return np.ascontiguousarray(a), np.ascontiguousarray(b), syn.upstream(g, n)


@pytest.mark.parametrize("angle,size", [(2, "small"), (2, "large"), (1, "small")])
def test_small_differences(enh, orc, angle, size):
    a, b, gm = near_pairs(angle, size)
    ra, rb = orc.mass_grad_def(a, b, gm)
    d = a[:, angle] - b[:, angle]
    for name in ("enh_pairs", "egh_pairs"):  # the second has no FP64 differences and declines instead
        ga, gb, ok, asked = _grads(enh, name, a, b, gm)
        for got, ref in ((ga, ra), (gb, rb)):
            ref = np.where(d == 0.0, 0.0, ref[:, angle])  # there the oracle's definition leaves 2^-110 of its terms
            assert np.all(np.abs(got[:, angle] - ref)[ok] <= TOL_F64 * np.abs(ref[ok]))
        if name == "enh_pairs":
            assert ok.all()
            assert not asked[np.abs(d) > 2.0 ** -11].any()
            assert not asked[np.min(np.abs(np.hstack([a[:, 1:3], b[:, 1:3]])), axis=1) > 2.0 ** -7].any()


@pytest.mark.parametrize("around", [2.0 ** -6.9, 2.0 ** -12, 0.0])
def test_nearly_collinear_massless_pairs(enh, around):
    """Both differences small and no mass to cover an error in them, between angles that the staged ones
    hold exactly and between angles that they do not: the gradient is right or the pair declined, never
    0 where the mass is not."""
    g = syn.rng(572)
    n = 20_000
    a, b = syn.ptetaphim(g, n), syn.ptetaphim(g, n)
    a[:, 3] = b[:, 3] = 0.0
    low = np.log2(around) if around else -60.0
    a[:, 1:3] = np.exp2(g.uniform(low, 1.5 if around > 2.0 ** -7 else -7.1, (n, 2))) * g.choice([-1.0, 1.0], (n, 2))
    b[:, 1:3] = a[:, 1:3] + 10.0 ** g.uniform(-17, -4, (n, 1)) * g.uniform(-1, 1, (n, 2))
    a, b, gm = np.ascontiguousarray(a), np.ascontiguousarray(b), syn.upstream(g, n)
    # closed form in FP64: m = 2 sqrt(pt pt S), whose relative error is that of S (no cancellation)
    de, dp = a[:, 1] - b[:, 1], a[:, 2] - b[:, 2]
    pp = a[:, 0] * b[:, 0]
    m = 2.0 * np.sqrt(pp * (np.sinh(0.5 * de) ** 2 + np.sin(0.5 * dp) ** 2))
    with np.errstate(invalid="ignore", divide="ignore"):
        ref = gm[:, None] * np.stack([0.5 * m / a[:, 0], pp * np.sinh(de) / m, pp * np.sin(dp) / m], axis=1)
    for name in ("enh_pairs", "egh_pairs"):
        ga, _, ok, _ = _grads(enh, name, a, b, gm)
        ok &= m > 0.0
        # d/dpt, d/dphi by themselves; d/deta besides the W term, which is 0 for massless legs
        assert np.all(np.abs(ga[:, :3] - ref)[ok] <= TOL_F64 * np.abs(ref)[ok])
        if name == "enh_pairs":
            assert ok[m > 2.0 ** -39 * np.maximum(a[:, 0], b[:, 0])].all()
