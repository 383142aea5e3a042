"""The FP64 pair mass at numbers of pairs around the lines between its launch shapes (one resident wave of
CTAs, two waves of six pairs per thread, 32 waves): every prefix of a sample has the sample's masses, bit
for bit."""
import pytest

import gvx_synth as syn
from helpers import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["soa", "aos"])
def test_prefixes(layout):
    import paper_2312_02756_gb300 as gvx
    torch = torch_cuda()
    g = syn.rng(571)
    wave = torch.cuda.get_device_properties(0).multi_processor_count * 8 * 128
    n = 40 * wave
    small = torch.as_tensor(syn.ptetaphim(g, 200_003)).cuda().t()
    a = small.repeat(1, n // small.shape[1] + 1)[:, :n].contiguous()
    b = a.roll(12345, 1).contiguous()
    if layout == "aos":
        a, b = a.t().contiguous(), b.t().contiguous()
    cut = (lambda v, k: v[:, :k]) if layout == "soa" else (lambda v, k: v[:k])
    want = gvx.invariant_mass(a, b, layout, layout)
    assert torch.isfinite(want).all()
    for k in (1, 127, 129, wave - 1, wave, wave + 1, 2 * wave + 5, 12 * wave - 769, 12 * wave, 12 * wave + 1,
              13 * wave + 77, 39 * wave - 1):
        assert torch.equal(gvx.invariant_mass(cut(a, k), cut(b, k), layout, layout), want[:k]), k
