"""The fused selection's 64-bit counts where one event has more pairs in one histogram slot than 32 bits
hold: 92,683 selected particles, 4,295,022,903 pairs (about 50 s on one block, nearly all of this test), and
events around it."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import torch_cuda

pytestmark = pytest.mark.gpu


def test_counts_of_an_event_beyond_32_bits():
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    sizes = np.array([5, 200, 92_683, 300, 64])
    off = np.concatenate([[0], np.cumsum(sizes)])
    p = syn.ptetaphim(syn.rng(591), int(off[-1]))
    p[:, 3] = 5.0  # every pair mass is at least 10
    counts, best_k, best_m = gvx.event_pair_select(t.as_tensor(p).cuda(), t.as_tensor(off).cuda(), 0.0, np.inf,
                                                   0.0, 10.0, 2, 10.0, layout="aos")
    assert counts.cpu().tolist() == [0, 0, 0, int(np.sum(sizes * (sizes - 1) // 2))]
    assert gvx.device_status() == 0
    assert (best_m.cpu().numpy() >= 10.0).all() and (best_k.cpu().numpy() >= 0).all()
