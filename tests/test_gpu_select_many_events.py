"""The fused selection where its grid grows beyond the CTAs that fit at once (more than 256 tiles of 32 events
per warp: from about 30 million events): the same counts and candidates as the halves in calls of their own."""
import pytest

from helpers import torch_cuda

pytestmark = pytest.mark.gpu


def test_more_events_than_one_wave_of_tiles():
    t = torch_cuda()
    import paper_2312_02756_gb300 as gvx
    sms = t.cuda.get_device_properties(0).multi_processor_count
    n = 256 * 8 * 3 * sms * 32 + 54_321
    g = t.Generator(device="cuda")
    g.manual_seed(613)
    off = t.zeros(n + 1, dtype=t.int64, device="cuda")
    t.cumsum(t.randint(0, 4, (n,), device="cuda", generator=g), 0, out=off[1:])
    u = t.rand(int(off[-1]), 4, dtype=t.float64, device="cuda", generator=g)
    p = u * t.tensor([100.0, 6.0, 6.28, 5.0], dtype=t.float64, device="cuda") - t.tensor(
        [0.0, 3.0, 3.14, 0.0], dtype=t.float64, device="cuda")
    del u
    cuts = (10.0, 2.5, 0.0, 200.0, 50, 91.1876)
    counts, best_k, best_m = gvx.event_pair_select(p, off, *cuts, layout="aos")
    h = n // 2
    parts = [gvx.event_pair_select(p[:int(off[h])], off[:h + 1].contiguous(), *cuts, layout="aos"),
             gvx.event_pair_select(p[int(off[h]):], (off[h:] - off[h]).contiguous(), *cuts, layout="aos")]
    assert gvx.device_status() == 0
    assert t.equal(counts, parts[0][0] + parts[1][0]) and int(counts.sum()) > n // 4
    assert t.equal(best_k, t.cat([q[1] for q in parts]))
    assert t.equal(best_m.nan_to_num(-1.0), t.cat([q[2] for q in parts]).nan_to_num(-1.0))
