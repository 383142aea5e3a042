"""Event sums and their gradients on the GPU component by component, for particles near eta = 0 or phi = 0:
events of one particle, and of several whose angles have one sign (so that no component cancels), as many
as a warp batch, a CTA and the general path take.  Tolerance: 1e-12 relative per component; what lies
below 2^-90 of the event's scale is compared absolutely."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda
from test_event_own_host import check, small_angles

pytestmark = pytest.mark.gpu


def _sizes(which, n):
    return np.full(n // which, which) if which else syn.rng(564).integers(0, 12, n // 6)


@pytest.mark.parametrize("which", [1, 3, 0, 40, 64, 100, 230])
def test_event_sums_by_component(orc, which):
    from test_gpu_jagged import _run
    torch_cuda()
    off = np.concatenate([[0], np.cumsum(_sizes(which, 6000))]).astype(np.int64)
    p = small_angles(int(off[-1]))
    p[:, 1:3] = np.abs(p[:, 1:3])
    for layout, sums_layout in (("aos", "soa"), ("soa", "aos")):
        _, _, sums = _run(p, off, layout, sums_layout)
        one = orc.to_cartesian_def(p)
        ref = np.add.reduceat(np.vstack([one, np.zeros((1, 4))]), off[:-1], axis=0)
        ref[np.diff(off) == 0] = 0.0
        check(sums, ref, ref[:, 3:], TOL_F64)


@pytest.mark.parametrize("k", range(4))
def test_sum_gradients_by_component(orc, k):
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    sizes = _sizes(0, 4000)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    po = np.concatenate([[0], np.cumsum(sizes * (sizes - 1) // 2)]).astype(np.int64)
    p = small_angles(int(off[-1]))
    gs = np.eye(4)[k] * syn.upstream(syn.rng(565), (len(sizes), 1))
    ref = orc.event_pairs_grad_def(p, off, np.zeros(int(po[-1])), gs)
    scale = np.repeat(np.abs(gs[:, k]), sizes) * np.maximum(p[:, 0], 1.0)
    for layout in ("aos", "soa"):
        x = t.as_tensor(p if layout == "aos" else np.ascontiguousarray(p.T)).cuda()
        got = gvx.event_pair_masses_bwd(x, t.as_tensor(off).cuda(), t.as_tensor(po).cuda(),
                                        t.zeros(int(po[-1]), dtype=t.float64, device="cuda"),
                                        t.as_tensor(gs).cuda(), layout, "aos").cpu().numpy()
        check(got if layout == "aos" else got.T, ref, scale[:, None], TOL_F64)
