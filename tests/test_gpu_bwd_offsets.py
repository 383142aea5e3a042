"""The jagged adjoint with malformed offsets: GVX_ERR_OFFSETS is recorded, the gradients of the events that the
wrong entry delimits are not written, and those of all others are, whatever tile they share."""
import numpy as np
import pytest

import gvx_synth as syn
from helpers import TOL_F64, torch_cuda

pytestmark = pytest.mark.gpu

OFFSETS = 6


@pytest.mark.parametrize("which", ["pair_offsets", "offsets", "last"])
@pytest.mark.parametrize("lam", [7.0, 25.0])
def test_only_the_events_with_wrong_offsets(orc, which, lam):
    from test_gpu_jagged_bwd import _err, _magnitudes
    t = torch_cuda()
    import ctypes
    import paper_2312_02756_gb300 as gvx
    from paper_2312_02756_gb300._lib import LV
    g = syn.rng(611)
    sizes = g.poisson(lam, 100)
    assert sizes[70] > 1 and sizes[71] > 1
    off = np.concatenate([[0], np.cumsum(sizes)])
    po = np.concatenate([[0], np.cumsum(sizes * (sizes - 1) // 2)])
    p = syn.ptetaphim(g, int(off[-1]))
    gm, gs = syn.upstream(g, int(po[-1])), syn.upstream(g, (100, 4))
    ref = orc.event_pairs_grad_def(p, off, gm, gs)
    wrong = {"pair_offsets": 37, "offsets": 71, "last": 100}[which]
    off2, po2 = off.copy(), po.copy()
    (off2 if which == "offsets" else po2)[wrong] += 1 if which != "last" else 10
    skipped = np.zeros(len(p), bool)
    skipped[off[wrong - 1]:off[min(wrong + 1, 100)]] = True
    x, go, gp = t.as_tensor(p).cuda(), t.as_tensor(gs).cuda(), t.full((len(p), 4), 7.5, dtype=t.float64).cuda()
    d_off, d_po, d_gm = t.as_tensor(off2).cuda(), t.as_tensor(po2).cuda(), t.as_tensor(gm).cuda()
    lib = gvx.load_library()
    lv = lambda v: LV((ctypes.c_void_p * 4)(v.data_ptr(), None, None, None), gvx.AOS)  # noqa: E731
    n_ws = lib.gvx_event_pair_masses_bwd_workspace(100)
    ws = t.empty(n_ws, dtype=t.uint8, device="cuda")
    assert lib.gvx_event_pair_masses_bwd(lv(x), d_off.data_ptr(), d_po.data_ptr(), 100, len(p), d_gm.data_ptr(),
                                         len(gm), lv(go), lv(gp), ws.data_ptr(), n_ws,
                                         ctypes.c_void_p(t.cuda.current_stream().cuda_stream)) == 0
    t.cuda.synchronize()
    assert gvx.device_status() == OFFSETS
    got = gp.cpu().numpy()
    assert np.all(got[skipped] == 7.5)
    assert np.max(_err(got, ref, _magnitudes(orc, p, off, gm, gs), p)[~skipped]) <= TOL_F64
