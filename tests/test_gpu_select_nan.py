"""The fused selection's best candidate where some pair masses are NaN (a particle without a direction): such a
pair is counted beyond the histogram's upper edge and is never the candidate while another pair of the
event has a mass, whichever part of the kernel takes the event (a warp, up to 128 particles; a staged
block, up to 256; the general path)."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [5, 40, 128, 129, 200, 256, 257, 400])
def test_pairs_without_a_mass(size):
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    n = 24
    g = syn.rng(601)
    p = syn.ptetaphim(g, n * size).reshape(n, size, 4)
    gone = np.zeros((n, size), bool)
    for e in range(n):  # one particle, then more of them; never of the first pair
        gone[e, 2 + g.permutation(size - 2)[:min(1 + e * size // 40, size - 3)]] = True
    p[gone, 2] = np.nan
    off = t.arange(n + 1, device="cuda") * size
    x = t.as_tensor(p.reshape(-1, 4)).cuda()
    pairs = size * (size - 1) // 2
    _, pm, _ = gvx.event_pair_masses(x, off, n * pairs, layout="aos")
    pm = pm.cpu().numpy().reshape(n, pairs)
    i, j = np.triu_indices(size, 1)
    assert np.array_equal(np.isnan(pm), gone[:, i] | gone[:, j])
    counts, best_k, best_m = gvx.event_pair_select(x, off, 0.0, np.inf, 0.0, 1e9, 3, 91.1876, layout="aos")
    best_k, best_m = best_k.cpu().numpy(), best_m.cpu().numpy()
    assert counts.cpu().numpy()[[0, -1]].tolist() == [0, int(np.isnan(pm).sum())] and int(counts.sum()) == pm.size
    least = np.nanmin(np.abs(pm - 91.1876), axis=1)
    got = pm[np.arange(n), best_k]
    assert np.all(np.abs(best_m - got) <= TOL_F64 * got)
    assert np.all(np.abs(got - 91.1876) <= least + TOL_F64 * got)
