"""The block replay's tile pipeline (operand tiles and accumulators taken in turn by several teams of warps) at every count of tiles of a
unit from 3 to 11, carried on from unit to unit by CTAs that replay several, with one and two code words, against the oracle, bit for
bit; at units with fewer tiles than their cluster has CTAs; and where large two-word tables leave room for one operand A buffer or for blocks
of 64 steps only, with units of a few blocks following one another on a CTA."""
import pytest

from cases import C
from parity import Case

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(ragged=True, head_dim=64)
many = base.scaled(batch=20, n_kv_heads=8, budget_lo=300, budget_hi=1400)  # 160 units
few = base.scaled(batch=3, n_kv_heads=2, budget_lo=40, budget_hi=1000)  # 6 units of up to 8 tiles, a CTA each
spread = base.scaled(batch=3, n_kv_heads=2, budget_lo=40, budget_hi=2000)  # 6 units of 11, 4 and 8 tiles in clusters of 8
large = C["throughput_batch"].scaled(batch=80, n_kv_heads=2, group_size=1, ragged=False, head_dim=64)  # 160 units
SHAPES = {
    "one_word": many.scaled(hash_bits=32),
    "two_words": many,
    "two_words_protected": many.scaled(n_sink=4, n_recent=10),
    "cluster_one_word": few.scaled(hash_bits=32),
    "cluster_two_words": few,
    "wide_cluster_one_word": spread.scaled(hash_bits=32),
    "wide_cluster_two_words": spread,
    "wide_cluster_two_words_protected": spread.scaled(n_sink=4, n_recent=10),
    "one_operand_buffer_over_sms": large.scaled(budget=8190, prompt_len=8400),
    "blocks_of_64_over_sms": large.scaled(budget=9830, prompt_len=9960),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_replay_tiles(name):
    if name.startswith("wide_cluster"):  # from 10 tiles on the widest cluster is the cheapest for six units
        tiles = [-(-int(b) // 128) for b in SHAPES[name].budgets()]
        assert max(tiles) >= 10 and min(tiles) < 8
    case = Case(SHAPES[name])
    case.prefill()
    case.compare_state()
