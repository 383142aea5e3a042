"""The jagged adjoint's batches and chunks at the sizes where they change hands (the events of
test_gpu_event_batches.py): events at and around the limits of a batch and of a chunk of pairs, even
and odd sizes (an even event's last row holds each of its pairs once), larger events, empty and
single ones, and the rare cases left to the second walk.  Checked against the oracle with the measure
and the tolerance of test_gpu_jagged_bwd.py."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda
from test_gpu_event_batches import COUNTS, _events
from test_gpu_jagged_bwd import _err, _gpu_bwd, _magnitudes, _n_pairs

pytestmark = pytest.mark.gpu

SIZES = dict(COUNTS, chunk_edge=[16, 17, 17, 18, 15, 12, 2, 2, 3, 64, 63, 62, 24, 33])


@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("which", list(SIZES))
def test_event_batches_bwd(orc, monkeypatch, which, extreme):
    torch_cuda()
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
    for layouts in (("aos", "soa", "soa"), ("soa", "aos", "aos")):
        for gs in (gsum, None):
            got = _gpu_bwd(p, off, gpm, gs, *layouts)
            ref = orc.event_pairs_grad_def(p, off, gpm, gs)
            mag = _magnitudes(orc, p, off, gpm, gs)
            assert np.isfinite(got).all()
            assert _err(got, ref, mag, p).max(initial=0.0) <= TOL_F64
