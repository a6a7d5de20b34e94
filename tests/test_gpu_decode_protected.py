"""Decode steps with protected windows where the kernel changes how it reads the slots' positions: copied beside a one-word table (256
threads up to 5120 slots, 512 threads from 8193), read from global memory where that leaves no room (5121 to 8192, above 12 288) and
beside two-word tables, with the last 16-byte vector cut short by the budget; and the same with the step's rows hashed in bulk."""
import pytest

from cases import C
from parity import Case

pytestmark = pytest.mark.gpu

base = C["llama3_8b_gqa"].scaled(batch=1, n_kv_heads=2, head_dim=64, n_sink=4, n_recent=10, decode_steps=6)


@pytest.mark.parametrize("budget,bits,group", [(5119, 32, 4), (5121, 32, 4), (6147, 16, 1), (8191, 32, 3), (8195, 32, 4), (12285, 24, 1), (12289, 32, 4),
                                               (3333, 64, 4), (9001, 40, 1)])
def test_protected_steps_at_the_edges_of_the_position_reads(budget, bits, group):
    case = Case(base.scaled(budget=budget, hash_bits=bits, group_size=group, prompt_len=budget + 9))
    case.prefill()
    case.decode(6, check_every=3)


@pytest.mark.parametrize("bits", [16, 64])
def test_protected_steps_with_the_rows_hashed_in_bulk(bits):
    w = C["throughput_batch"].scaled(batch=228, group_size=8, head_dim=64, hash_bits=bits, budget_lo=40, budget_hi=64, prompt_factor=1,
                                     n_sink=4, n_recent=10, decode_steps=4)
    assert w.n_units * (w.group_size + 1) >= 16384
    case = Case(w)
    case.prefill()
    case.decode(4, check_every=2)
