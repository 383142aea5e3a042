"""The jagged adjoint on the GPU where a pair's one angle difference is small and the other is not: events
of two particles with the upstream gradient on their mass, d/dphi (d/deta) by itself, and the same pairs
among other particles.  Tolerance: 1e-12 relative, the adjoint's gate."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda
from test_event_grad_near_host import near_pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("others", [0, 5])
@pytest.mark.parametrize("angle,size", [(2, "small"), (2, "large"), (1, "small")])
def test_small_differences(orc, angle, size, others):
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    a, b, g = near_pairs(angle, size, 4000)
    n, k = len(a), 2 + others
    p = np.empty((n, k, 4))
    p[:, 0], p[:, 1] = a, b
    p[:, 2:] = syn.ptetaphim(syn.rng(573), n * others).reshape(n, others, 4)
    p = p.reshape(-1, 4)
    off = np.arange(n + 1) * k
    pairs = k * (k - 1) // 2
    gm = np.zeros((n, pairs))
    gm[:, 0] = g  # the pair (0, 1) alone
    ra, rb = orc.mass_grad_def(a, b, g)
    d = a[:, angle] - b[:, angle]
    for layout in ("aos", "soa"):
        x = t.as_tensor(p if layout == "aos" else np.ascontiguousarray(p.T)).cuda()
        got = gvx.event_pair_masses_bwd(x, t.as_tensor(off).cuda(), t.as_tensor(np.arange(n + 1) * pairs).cuda(),
                                        t.as_tensor(gm.reshape(-1)).cuda(), layout=layout).cpu().numpy()
        got = (got if layout == "aos" else got.T).reshape(n, k, 4)
        for leg, ref in ((0, ra), (1, rb)):
            ref = np.where(d == 0.0, 0.0, ref[:, angle])
            assert np.all(np.abs(got[:, leg, angle] - ref) <= TOL_F64 * np.abs(ref))
        assert not got[:, 2:].any()
