"""The jagged adjoint's batches and chunks at the sizes where they change hands (the events of
test_gpu_event_batches.py): events at and around the limits of a batch and of a chunk of pairs, even
and odd sizes (an even event's last row holds each of its pairs once), larger events, empty and
single ones, and the rare cases left to the second launch; and numbers of events on both sides of the
lines between its tile shapes.  Checked against the oracle with the measure and the tolerance of
test_gpu_jagged_bwd.py."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda
from test_gpu_event_batches import COUNTS, _events
from test_gpu_jagged_bwd import _err, _gpu_bwd, _magnitudes, _n_pairs

pytestmark = pytest.mark.gpu

SIZES = dict(COUNTS, chunk_edge=[16, 17, 17, 18, 15, 12, 2, 2, 3, 64, 63, 62, 24, 33],
             staged_edge=[65, 8, 129], many=np.diff(syn.jagged_offsets(syn.rng(411), 300, lam=11.0)))


def _case(which, extreme, monkeypatch):
    monkeypatch.setitem(COUNTS, which, SIZES[which])
    off, p = _events(which, extreme)
    if extreme and len(p) > 5:
        p[4::37, 0] = 0.0  # pt = 0 with a mass
    g = syn.rng(431)
    gpm, gsum = syn.upstream(g, _n_pairs(off)), syn.upstream(g, (len(off) - 1, 4))
    if extreme:
        gpm[::101] *= 1e9
        gpm[5::103] = 0.0
        gsum[2::13] *= 1e-120
    return off, p, gpm, gsum


@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("which", list(SIZES))
def test_event_batches_bwd(orc, monkeypatch, which, extreme):
    torch_cuda()
    off, p, gpm, gsum = _case(which, extreme, monkeypatch)
    for gs in (gsum, None):
        ref = orc.event_pairs_grad_def(p, off, gpm, gs)
        mag = _magnitudes(orc, p, off, gpm, gs)
        for layouts in (("aos", "soa", "soa"), ("soa", "aos", "aos")):
            got = _gpu_bwd(p, off, gpm, gs, *layouts)
            assert np.isfinite(got).all()
            assert _err(got, ref, mag, p).max(initial=0.0) <= TOL_F64


@pytest.mark.parametrize("extreme", [False, True])
def test_event_numbers_bwd(orc, monkeypatch, extreme):
    """300 events over and over, up to 393,000 of them: every copy has the gradients of the first."""
    torch_cuda()
    off, p, gpm, gsum = _case("many", extreme, monkeypatch)
    ref = orc.event_pairs_grad_def(p, off, gpm, gsum)
    mag = _magnitudes(orc, p, off, gpm, gsum)
    for copies in (100, 320, 340, 640, 660, 1290, 1310):
        big = np.concatenate([[0], np.cumsum(np.tile(np.diff(off), copies))]).astype(np.int64)
        got = _gpu_bwd(np.tile(p, (copies, 1)), big, np.tile(gpm, copies), np.tile(gsum, (copies, 1)))
        got = got.reshape(copies, len(p), 4)
        assert np.isfinite(got).all()
        for k in sorted({0, 1, copies // 2, copies - 1}):
            assert _err(got[k], ref, mag, p).max() <= TOL_F64, (copies, k)
        spread = np.abs(got - got[0]).max(axis=0)  # the rest against the first
        assert _err(spread, np.zeros_like(p), mag, p).max() <= 2 * TOL_F64, copies
