"""Attention over the cache at the edges of its 32-slot groups and of the split over a cluster, for both head sizes of the
tensor-core kernel: fill levels inside a group, budgets from one group to several CTAs' worth, one unit and more units than
SMs. Slots beyond the fill level hold NaN, which must not reach the output."""
import pytest
import torch

from paper_2412_16187_b200 import HashEvictCache, device_error_count

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [64, 128])
@pytest.mark.parametrize("batch,heads,group,budget", [(1, 1, 4, 9830), (1, 8, 8, 4096), (2, 4, 1, 1000), (1, 32, 3, 300), (50, 4, 4, 100)])
def test_attend_split(dim, batch, heads, group, budget):
    g = torch.Generator(device="cuda").manual_seed(budget + dim)
    c = HashEvictCache(batch, heads, group, dim, 32, [budget] * batch, torch.randn(dim, 32))
    shape = tuple(c.k_cache.shape)
    c.k_cache.copy_(torch.randn(shape, device="cuda", generator=g))
    c.v_cache.copy_(torch.randn(shape, device="cuda", generator=g))
    fill = torch.randint(0, budget + 1, (batch, heads), device="cuda", generator=g, dtype=torch.int32)
    fill.view(-1)[0] = budget
    fill.view(-1)[-1] = min(33, budget) if batch * heads > 1 else budget - 7
    c.fill.copy_(fill)
    valid = torch.arange(shape[2], device="cuda").view(1, 1, -1) < fill.unsqueeze(2)
    c.k_cache.masked_fill_(~valid.unsqueeze(3), float("nan"))
    c.v_cache.masked_fill_(~valid.unsqueeze(3), float("nan"))
    q = torch.randn(batch, heads * group, dim, device="cuda", generator=g).to(torch.bfloat16)
    out = c.attend(q)
    k = torch.nan_to_num(c.k_cache).double()
    v = torch.nan_to_num(c.v_cache).double()
    s = torch.einsum("bhgd,bhjd->bhgj", q.view(batch, heads, group, dim).double(), k) / dim ** 0.5
    w = torch.nan_to_num(torch.softmax(s.masked_fill(~valid.unsqueeze(2), float("-inf")), dim=3))
    want = torch.einsum("bhgj,bhjd->bhgd", w, v).view(batch, heads * group, dim)
    assert (out.double() - want).abs().max().item() < 2e-5 * v.abs().max().item()
    assert device_error_count() == 0
