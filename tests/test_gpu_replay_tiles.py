"""The block replay's tile pipeline (operand tiles and accumulators taken in turn by several teams of warps) at every count of tiles of a
unit from 3 to 11, carried on from unit to unit by CTAs that replay several, with one and two code words, against the oracle, bit for
bit; and at units with fewer tiles than their cluster has CTAs."""
import pytest

from cases import C
from parity import Case

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(ragged=True, head_dim=64)
many = base.scaled(batch=20, n_kv_heads=8, budget_lo=300, budget_hi=1400)  # 160 units
few = base.scaled(batch=3, n_kv_heads=2, budget_lo=40, budget_hi=1000)
SHAPES = {
    "one_word": many.scaled(hash_bits=32),
    "two_words": many,
    "two_words_protected": many.scaled(n_sink=4, n_recent=10),
    "cluster_one_word": few.scaled(hash_bits=32),
    "cluster_two_words": few,
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_replay_tiles(name):
    case = Case(SHAPES[name])
    case.prefill()
    case.compare_state()
