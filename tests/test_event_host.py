"""CPU checks of the event kernels' staged pair (csrc/event_lc.cuh: fixed-point angles, the turn
in d_phi, the light-cone sum of two staged particles), compiled for the host from the same source,
against the binary128 oracle.

Tolerance: 2^-42 relative, the bound of the float-float route (mass_lc.cuh); the fixed-point angles
add at most 2^-47 where S >= 2^-22, and a pair below that has to be declined."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import gvx_synth as syn
from helpers import edge_pairs

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def evh(tmp_path_factory):
    from paper_2312_02756_gb300 import gen_tables
    out = str(tmp_path_factory.mktemp("evh"))
    gen_tables.write(os.path.join(out, "gvx_tables.inc"))
    lib = os.path.join(out, "evh.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + out,
                    os.path.join(HERE, "event_harness.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _turned(n):
    """Pairs on either side of phi = +-pi, from 1e-6 to 0.5 apart, and pairs close in both angles."""
    g = syn.rng(401)
    a, b = syn.ptetaphim(g, n), syn.ptetaphim(g, n)
    d = 10.0 ** g.uniform(-6, -0.3, n)
    f = g.uniform(0.0, 1.0, n)
    a[:, 2], b[:, 2] = np.pi - f * d, -np.pi + (1 - f) * d
    b[::2, 1] = a[::2, 1] + 10.0 ** g.uniform(-6, -1, n)[::2]
    b[::4, 2] = a[::4, 2] - d[::4]
    a[::3], b[::3] = b[::3].copy(), a[::3].copy()
    return a, b


@pytest.mark.parametrize("which", ["plain", "light", "turned", "edge"])
def test_staged_pair_against_oracle(evh, orc, which):
    n = 100_000
    a, b = {"plain": lambda: (syn.ptetaphim(syn.rng(0), n), syn.ptetaphim(syn.rng(7), n)),
            "light": lambda: (syn.ptetaphim_light_mix(syn.rng(2), n), syn.ptetaphim_light_mix(syn.rng(3), n)),
            "turned": lambda: _turned(n), "edge": edge_pairs}[which]()
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    m, ok = np.empty(len(a)), np.empty(len(a), np.uint8)
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    evh.evh_pairs(p(a), p(b), ctypes.c_int64(len(a)), p(m), p(ok))
    ok = ok.astype(bool)
    ref = orc.mass_def(a, b, nthreads=8)
    assert np.all(np.abs(m - ref)[ok] <= 2.0 ** -42 * ref[ok])
    dphi = np.abs(a[:, 2] - b[:, 2])
    dphi = np.minimum(dphi, 2 * np.pi - dphi)
    s = np.sinh(0.5 * (a[:, 1] - b[:, 1])) ** 2 + np.sin(0.5 * dphi) ** 2
    assert not ok[s < 0.9 * 2.0 ** -22].any()
    if which != "edge":
        assert ok[s > 1.1 * 2.0 ** -22].all()
