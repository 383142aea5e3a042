"""The event kernels' batches at the sizes where they change hands: events at and around the
limits of a warp batch, of an event staged by a CTA and beyond it, runs of empty and single events,
few events and many, particles outside the float-float domain and pairs close in both angles.
Checked against the oracle with the tolerances of test_gpu_jagged.py and test_gpu_select.py."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import torch_cuda

pytestmark = pytest.mark.gpu

COUNTS = {
    "one": [1], "empty": [0] * 70, "pair": [2], "few": [3, 0, 9, 1, 5, 2, 7],
    "batch_edge": [64, 1, 63, 64, 65, 32, 32, 33, 31, 0, 64],
    "staged_edge": [223, 8, 224, 9, 225, 10, 128, 129, 255, 11, 256, 257],
    "small": [0, 1, 2] * 60 + [40] + [1] * 90,
    "many": None,
}


def _events(which, extreme):
    g = syn.rng(410)
    counts = COUNTS[which]
    if counts is None:
        counts = np.diff(syn.jagged_offsets(g, 5001, lam=11.0))
    off = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    p = syn.ptetaphim(g, int(off[-1]))
    if extreme:
        p[3::41, 1] = 12.5             # |eta| >= 8
        p[5::53] = [0.0, 0.3, 0.2, 0.0]  # a zero vector
        p[7::29, 2] = np.pi            # the ends of phi
        p[8::31, 2] = -np.pi
        k = np.arange(11, len(p), 17)  # next to the particle before, in both angles
        p[k, 1:3] = p[k - 1, 1:3]
        p[k[1::2], 1] += 1e-5
    return off, p


@pytest.mark.parametrize("extreme", [False, True])
@pytest.mark.parametrize("which", list(COUNTS))
def test_event_batches(orc, which, extreme):
    from test_gpu_jagged import _check, _run
    torch_cuda()
    off, p = _events(which, extreme)
    for layout, sums_layout in (("aos", "soa"), ("soa", "aos")):
        po, pm, sums = _run(p, off, layout, sums_layout)
        _check(orc, p, off, po, pm, sums)


@pytest.mark.parametrize("pt_min,eta_max", [(0.0, np.inf), (20.0, 2.5), (30.0, 0.7), (2000.0, 2.5)])
@pytest.mark.parametrize("which", list(COUNTS))
def test_select_batches(orc, which, pt_min, eta_max):
    from test_gpu_select import _check, _run
    torch_cuda()
    off, p = _events(which, True)
    cuts = dict(pt_min=pt_min, eta_max=eta_max, lo=5.0, hi=350.0, n_bins=137, target=91.1876)
    for layout in ("aos", "soa"):
        c, bk, bm = _run(p, off, layout, **cuts)
        _check(orc, p, off, c, bk, bm, **cuts)


def test_select_cuts_on_bits():
    """The cuts' integer comparisons take what the FP64 ones take: NaN fails either cut, -0 passes a
    threshold of 0, infinities and negative thresholds order as numbers."""
    import paper_2312_02756_gb300 as gvx
    torch = torch_cuda()
    pts = np.array([-0.0, 0.0, 5e-324, -1.0, 1.0, np.inf, -np.inf, np.nan, 20.0, np.nextafter(20.0, 0)])
    etas = np.array([0.0, -0.0, 2.5, -2.5, np.nextafter(2.5, 9), np.inf, -np.inf, np.nan, -1.0])
    p = np.array([[x, e, 0.1, 1.0] for x in pts for e in etas])
    off = torch.arange(0, 2 * len(p) + 1, 2).cuda()
    two = torch.as_tensor(np.repeat(p, 2, axis=0)).cuda()
    for pt_min in (0.0, -0.0, 20.0, -1.0, np.inf, -np.inf, np.nan):
        for eta_max in (2.5, 0.0, np.inf, -1.0, np.nan):
            counts, _, _ = gvx.event_pair_select(two, off, pt_min, eta_max, 0.0, 10.0, 4, 1.0)
            want = int(np.sum((p[:, 0] >= pt_min) & (np.abs(p[:, 1]) <= eta_max)))
            assert int(counts.sum()) == want, (pt_min, eta_max)
    assert gvx.device_status() == 0
