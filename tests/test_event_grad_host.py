"""CPU checks of the jagged adjoint's pair and particle arithmetic (csrc/event_lc_grad.cuh), compiled
for the host from the same source, against the binary128 oracle.

Error measure: the largest component error of a leg's gradient weighted by max(|x_k|, 1), relative to
the same weighting of the summed magnitudes of its contributions.  Tolerance 1e-12, the adjoint's gate on the GPU."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def egh(tmp_path_factory):
    from paper_2312_02756_gb300 import gen_tables
    out = str(tmp_path_factory.mktemp("egh"))
    gen_tables.write(os.path.join(out, "gvx_tables.inc"))
    lib = os.path.join(out, "egh.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + out,
                    os.path.join(HERE, "event_grad_harness.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _err(got, ref, x, mag=None):
    s = np.maximum(np.abs(x), 1.0)
    mag = np.abs(ref) if mag is None else mag
    return np.max(np.abs(got - ref) * s, axis=1) / np.maximum(np.sum(mag * s, axis=1), 1e-300)


@pytest.mark.parametrize("which", ["plain", "light", "turned", "soft", "small_g"])
def test_pair_gradients_against_oracle(egh, orc, which):
    n = 50_000
    g = syn.rng(501)
    mk = syn.ptetaphim_light_mix if which == "light" else syn.ptetaphim
    a, b = mk(g, n), mk(g, n)
    gm = syn.upstream(g, n)
    if which == "turned":
        d = 10.0 ** g.uniform(-3, -0.3, n)
        a[:, 2], b[:, 2] = np.pi - 0.3 * d, -np.pi + 0.7 * d
        a[::2], b[::2] = b[::2].copy(), a[::2].copy()
    if which == "soft":
        b[:, [0, 3]] *= 2.0 ** g.uniform(-25, 0, (n, 1))
    if which == "small_g":
        gm *= 2.0 ** g.uniform(-40, 14, n)
    a, b, gm = (np.ascontiguousarray(v) for v in (a, b, gm))
    ga, gb, ok = np.empty_like(a), np.empty_like(a), np.empty(n, np.uint8)
    egh.egh_pairs(_p(a), _p(b), _p(gm), ctypes.c_int64(n), _p(ga), _p(gb), _p(ok))
    ok = ok.astype(bool)
    assert ok.mean() > 0.999
    ra, rb = orc.mass_grad_def(a, b, gm)
    assert max(_err(ga[ok], ra[ok], a[ok]).max(), _err(gb[ok], rb[ok], b[ok]).max()) <= TOL_F64


def test_sum_gradients_against_oracle(egh, orc):
    n = 20_000
    g = syn.rng(502)
    p, gs = syn.ptetaphim(g, n), syn.upstream(g, (n, 4))
    p[::7, 3] = 0.0
    p[::11, 1:3] *= 1e-6
    gs *= 2.0 ** g.uniform(-280, 280, (n, 1))
    out, ok = np.empty_like(p), np.empty(n, np.uint8)
    egh.egh_sums(_p(p), _p(gs), ctypes.c_int64(n), _p(out), _p(ok))
    assert ok.all()
    off = np.arange(n + 1)
    ref = orc.event_pairs_grad_def(p, off, np.zeros(0), gs)
    mag = sum(np.abs(orc.event_pairs_grad_def(p, off, np.zeros(0), np.eye(4)[k] * gs)) for k in range(4))
    assert _err(out, ref, p, mag).max() <= TOL_F64
