"""CPU checks of a staged particle's own terms (csrc/event_lc.cuh, event_lc_grad.cuh), compiled for the
host from the same source: its Cartesian components and J^T gs of it, every component by itself, for
angles from the ordinary down to 1e-30 and 0.  Tolerance per component: 2^-42 relative, a few of the
float-float steps' 2^-46; for J^T gs, a chain of up to six of them, 1e-12, the adjoint's gate.
Components below 2^-90 of the particle's scale are compared absolutely."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64

HERE = os.path.dirname(os.path.abspath(__file__))
TOL = 2.0 ** -42


@pytest.fixture(scope="module")
def eoh(tmp_path_factory):
    from paper_2312_02756_gb300 import gen_tables
    out = str(tmp_path_factory.mktemp("eoh"))
    gen_tables.write(os.path.join(out, "gvx_tables.inc"))
    lib = os.path.join(out, "eoh.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + out,
                    os.path.join(HERE, "event_own_harness.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def small_angles(n):
    """Particles whose eta and phi are log-uniform from 1 down to 1e-30, of either sign, some exactly 0
    and some at the steps of the reduction (2^-12, 2^-9)."""
    g = syn.rng(561)
    p = syn.ptetaphim(g, n)
    p[:, 1:3] = 10.0 ** g.uniform(-30, 0, (n, 2)) * g.choice([-1.0, 1.0], (n, 2))
    p[::2, 1:3] = 10.0 ** g.uniform(-6, 0, (len(p[::2]), 2)) * g.choice([-1.0, 1.0], (len(p[::2]), 2))
    p[::17, 1] = p[3::19, 2] = 0.0
    p[5::23, 1] = -2.0 ** -12
    p[7::23, 2] = np.nextafter(2.0 ** -12, 0.0)
    p[9::23, 1] = 2.0 ** -9
    p[11::13, 3] = 0.0
    return p


def check(got, ref, scale, tol=TOL):
    assert np.all(np.abs(got - ref) <= tol * np.abs(ref) + 2.0 ** -90 * scale)


def test_components(eoh, orc):
    p = np.ascontiguousarray(small_angles(40_000))
    out, ok = np.empty_like(p), np.empty(len(p), np.uint8)
    eoh.eoh_cart(_p(p), ctypes.c_int64(len(p)), _p(out), _p(ok))
    assert ok.all()
    check(out, orc.to_cartesian_def(p), np.maximum(p[:, 0], p[:, 3])[:, None])


@pytest.mark.parametrize("k", range(4))
def test_sum_gradients_by_component(eoh, orc, k):
    """One upstream component at a time, so that every entry of the result is one product."""
    p = np.ascontiguousarray(small_angles(20_000))
    gs = np.ascontiguousarray(np.eye(4)[k] * syn.upstream(syn.rng(562), (len(p), 1)))
    out, ok = np.empty_like(p), np.empty(len(p), np.uint8)
    eoh.eoh_sums(_p(p), _p(gs), ctypes.c_int64(len(p)), _p(out), _p(ok))
    assert ok.all()
    ref = orc.event_pairs_grad_def(p, np.arange(len(p) + 1), np.zeros(0), gs)
    check(out, ref, (np.abs(gs[:, k]) * np.maximum(p[:, 0], 1.0))[:, None], TOL_F64)
