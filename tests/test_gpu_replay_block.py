"""The block replay kernel against the oracle at the edges of its tiles, of its block sizes and of its shared-memory
layouts: budgets around 128-slot tiles and around the budgets where the block gets longer, every group size's operand
scaling, one unit spread over a whole cluster, more units than clusters, and a two-word table that leaves room for one
operand A buffer only."""
import pytest

from cases import C
from parity import Case

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(batch=1, n_kv_heads=2, ragged=False)
SHAPES = {
    **{f"budget_{c}": base.scaled(budget=c, prompt_len=c + 300) for c in (1, 31, 127, 128, 129, 256, 1535, 1537)},
    **{f"group_{g}": base.scaled(group_size=g, hash_bits=b, budget=390, prompt_len=900) for g, b in ((1, 32), (2, 24), (5, 64), (6, 32), (8, 64))},
    "one_unit_cluster": base.scaled(n_kv_heads=1, hash_bits=32, budget=9830, prompt_len=10300),
    "one_unit_cluster_protected": base.scaled(n_kv_heads=1, hash_bits=32, budget=5000, prompt_len=5400, n_sink=4, n_recent=100),
    "two_words_large": base.scaled(n_kv_heads=1, budget=8190, prompt_len=8600),
    "two_words_largest": base.scaled(n_kv_heads=1, budget=9830, prompt_len=10200),
    "units_over_clusters": base.scaled(batch=4, n_kv_heads=25, hash_bits=32, ragged=True, budget_lo=300, budget_hi=2600, head_dim=64),
    "units_over_sms": base.scaled(batch=10, n_kv_heads=16, ragged=True, budget_lo=200, budget_hi=500, head_dim=64),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_replay_block(name):
    case = Case(SHAPES[name])
    case.prefill()
    case.compare_state()
