"""CPU checks of the FP64 pair-mass adjoint (csrc/mass_lc_grad.cuh), compiled for the host from the same
source, for legs at and near eta = 0, where d/deta carries sinh(eta) as a factor: the error measure and
tolerance of the adjoint (each component weighted by max(|x|, 1), 1e-12), for d/deta by itself."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64
from test_ff_host import _mass_grad_lc, ffh  # noqa: F401 (fixture)


def small_eta(which, n=20_000):
    g = syn.rng(581)
    a, b = syn.ptetaphim(g, n), syn.ptetaphim(g, n)
    z = {"zero": np.zeros(n), "2^-30": 2.0 ** -30 * g.uniform(-1.5, 1.5, n),
         "tiny": 10.0 ** g.uniform(-40, -9, n) * g.choice([-1.0, 1.0], n)}[which]
    a[:, 1] = z
    b[::3, 1] = -z[::3]
    return np.ascontiguousarray(a), np.ascontiguousarray(b), syn.upstream(g, n)


def check_deta(a, b, gm, ga, gb, ra, rb):
    """|error of d/deta| against its two terms' magnitudes, the W term's and the sinh(d_eta) term's."""
    e = [np.hypot(v[:, 0] * np.cosh(v[:, 1]), v[:, 3]) for v in (a, b)]
    m = np.sqrt(np.abs((e[0] + e[1]) ** 2 - (a[:, 0] * np.sinh(a[:, 1]) + b[:, 0] * np.sinh(b[:, 1])) ** 2
                       - a[:, 0] ** 2 - b[:, 0] ** 2 - 2 * a[:, 0] * b[:, 0] * np.cos(a[:, 2] - b[:, 2])))
    w = np.abs(gm / m) * (e[0] * e[1] + a[:, 0] * b[:, 0])
    mag = w * (np.abs(np.sinh(a[:, 1])) + np.abs(np.sinh(b[:, 1])) + np.abs(np.sinh(a[:, 1] - b[:, 1])))
    for got, ref in ((ga, ra), (gb, rb)):
        assert np.all(np.abs(got - ref)[:, 1] <= TOL_F64 * mag + 1e-30 * w)


@pytest.mark.parametrize("which", ["zero", "2^-30", "tiny"])
def test_mass_adjoint_near_eta_0(ffh, orc, which):  # noqa: F811
    a, b, gm = small_eta(which)
    ga, gb, ok = _mass_grad_lc(ffh, a, b, gm)
    assert ok.all()
    ra, rb = orc.mass_grad_def(a, b, gm)
    check_deta(a, b, gm, ga, gb, ra, rb)
