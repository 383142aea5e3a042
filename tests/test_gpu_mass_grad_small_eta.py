"""The FP64 pair-mass adjoint on the GPU for legs at and near eta = 0: through autograd, and where the jagged
adjoint takes it for the pairs of an event too large to stage.  Tolerances of
test_mass_grad_small_eta_host.py."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import dev, host, torch_cuda
from test_mass_grad_small_eta_host import check_deta, small_eta

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("which", ["zero", "2^-30", "tiny"])
def test_mass_adjoint_near_eta_0(orc, which, layout):
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    a, b, gm = small_eta(which)
    x, y = (dev(v, layout).requires_grad_(True) for v in (a, b))
    gvx.invariant_mass(x, y, layout, layout).backward(t.as_tensor(gm).cuda())
    check_deta(a, b, gm, host(x.grad, layout), host(y.grad, layout), *orc.mass_grad_def(a, b, gm))


def test_large_events_near_eta_0(orc):
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    a, b, g = small_eta("tiny", 200)
    n, k = len(a), 72
    p = np.empty((n, k, 4))
    p[:, 0], p[:, 1] = a, b
    p[:, 2:] = syn.ptetaphim(syn.rng(583), n * (k - 2)).reshape(n, k - 2, 4)
    pairs = k * (k - 1) // 2
    gm = np.zeros((n, pairs))
    gm[:, 0] = g  # the pair (0, 1) alone
    got = gvx.event_pair_masses_bwd(t.as_tensor(p.reshape(-1, 4)).cuda(), t.arange(n + 1, device="cuda") * k,
                                    t.arange(n + 1, device="cuda") * pairs, t.as_tensor(gm.reshape(-1)).cuda(),
                                    layout="aos").cpu().numpy().reshape(n, k, 4)
    check_deta(a, b, g, got[:, 0], got[:, 1], *orc.mass_grad_def(a, b, g))
