"""Decode calls of many sequences: the budgets of up to 792 travel in the kernel parameters, and with inputs staged ahead the order
that units are dealt in (up to 396 sequences with their budgets); beyond, and without a host mirror, budgets are read on the device.
Victims and state against the oracle on both sides of the limits, and the dealing by its effect on the time."""
import pytest
import torch

from cases import C
from paper_2412_16187_b200 import HashEvictCache
from parity import Case

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(head_dim=64, budget_lo=5, budget_hi=90, decode_steps=3)


@pytest.mark.parametrize("early", [False, True])
@pytest.mark.parametrize("batch,heads,bits", [(256, 2, 64), (257, 2, 64), (296, 2, 24), (300, 1, 64), (396, 1, 64), (397, 1, 32), (592, 1, 32), (792, 1, 64), (793, 1, 32), (1024, 1, 64)])
def test_many_ragged_sequences_match_the_oracle(batch, heads, bits, early):
    case = Case(base.scaled(batch=batch, n_kv_heads=heads, hash_bits=bits, ragged=True), early_inputs=early)
    case.prefill()
    case.decode(3, check_every=3)


def test_many_packed_sequences_match_the_oracle():
    case = Case(base.scaled(batch=300, n_kv_heads=1, hash_bits=16, ragged=True), packed_codes=True)
    case.prefill()
    case.decode(3, check_every=3)


def test_budgets_beyond_16_bits():
    """Byte-packed tables hold more than 65 535 slots; their budgets travel as 32-bit values."""
    batch, dim, bits, budgets = 3, 64, 8, [70000, 65535, 65536]
    g = torch.Generator(device="cuda").manual_seed(2)
    W = torch.randn(dim, bits)
    q = torch.randn(batch, 4, dim, device="cuda", generator=g).to(torch.bfloat16)
    k = torch.randn(batch, 1, dim, device="cuda", generator=g).to(torch.bfloat16)
    codes = torch.randint(0, 256, (batch, 1, 70000, 1), device="cuda", generator=g, dtype=torch.uint8)

    def step(mirror):
        c = HashEvictCache(batch, 1, 4, dim, bits, budgets, W, packed_codes=True, host_budget_mirror=mirror)
        c.codes_storage[:, :, :70000].copy_(codes)
        c.fill.copy_(c.budget[:, None])
        c.next_pos.copy_(c.fill)
        c.pos.copy_(torch.arange(c.Cmax, device="cuda").expand_as(c.pos))
        victims = torch.stack([c.decode_step(q, k, k) for _ in range(3)])
        return victims, c.codes_storage, c.scores, c.pos

    for name, x, y in zip(("victims", "codes", "scores", "pos"), step(True), step(False)):
        assert torch.equal(x, y), name


def test_units_of_many_sequences_are_dealt_by_budget():
    """592 sequences of one unit on 148 SMs. In sequence order a CTA's four units are ranks i, 295 - i, 296 + i, 591 - i; the long
    budgets sit where that order gives all of them to eight CTAs. Dealt by budget no CTA has two, and the call is shorter."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    batch, dim, bits = 4 * sms, 128, 64
    budgets = torch.full((batch,), 64)
    for i in range(8):
        for rank in (i, 2 * sms - 1 - i, 2 * sms + i, 4 * sms - 1 - i):
            budgets[rank] = 4096
    g = torch.Generator(device="cuda").manual_seed(1)
    q = torch.randn(batch, 4, dim, device="cuda", generator=g).to(torch.bfloat16)
    k = torch.randn(batch, 1, dim, device="cuda", generator=g).to(torch.bfloat16)

    def time(mirror):
        c = HashEvictCache(batch, 1, 4, dim, bits, budgets, torch.randn(dim, bits), early_inputs=True, host_budget_mirror=mirror)
        c.fill.copy_(c.budget[:, None])
        c.next_pos.copy_(c.fill)
        c.pos.copy_(torch.arange(c.Cmax, device="cuda").expand_as(c.pos))
        out = torch.empty((batch, 1), dtype=torch.int32, device="cuda")
        c.decode_step(q, k, k, victim_out=out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            for _ in range(64):
                c.decode_step(q, k, k, victim_out=out)
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            graph.replay()
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times)[4]

    in_order, by_budget = time(False), time(True)
    assert by_budget < 0.9 * in_order, (by_budget, in_order)
