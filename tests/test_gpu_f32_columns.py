"""FP32 pair masses of columns: the kernel that takes four pairs per thread (all columns on 16-byte
boundaries) against the one that takes any alignment, at every remainder of four, few pairs and
many, and with a single column off its boundary.

Tolerance: 2^-21 relative; both round every operation of the same formulas to float, about 20 of
them of relative error 2^-24 each."""
import pytest

import gvx_synth as syn
from helpers import torch_cuda

pytestmark = pytest.mark.gpu


def _columns(torch, rows, shift):
    """(4, n) columns whose rows start `shift` elements off a 16-byte boundary."""
    n = rows.shape[1]
    stride = (n + shift + 3) // 4 * 4 + 4
    store = torch.full((4 * stride + 4,), float("nan"), dtype=torch.float32, device="cuda")
    out = torch.as_strided(store, (4, n), (stride, 1), shift)
    out.copy_(rows)
    return out


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 255, 1024, 1025, 4099, 311 * 1024 + 2])
def test_f32_columns(n):
    import paper_2312_02756_gb300 as gvx
    torch = torch_cuda()
    g = syn.rng(561)
    a, b = (torch.as_tensor(syn.to_f32(syn.ptetaphim_light_mix(g, n))).cuda().t() for _ in range(2))
    want = gvx.invariant_mass(_columns(torch, a, 1), _columns(torch, b, 3), "soa", "soa")
    for sa, sb in ((0, 0), (0, 2), (1, 0)):
        got = gvx.invariant_mass(_columns(torch, a, sa), _columns(torch, b, sb), "soa", "soa")
        assert torch.isfinite(got).all()
        assert ((got - want).abs() <= 2.0 ** -21 * want).all()
