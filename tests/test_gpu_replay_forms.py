"""The block replay at both ends of what its 16-bit tile keys hold and on both sides of where its owner table changes from words to
bytes: the largest ranks (odd groups of two-word codes, groups of eight), codes of a few bits (most keys tie, and recent tokens hold
best slots), tables just within and just beyond the word table's limit, and few-bit codes of more units than SMs, against the
oracle, bit for bit."""
import pytest

from cases import C
from parity import Case

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(batch=1, n_kv_heads=2, ragged=False)
SHAPES = {
    "group_7_b64": base.scaled(group_size=7, budget=257, prompt_len=700),
    "group_3_b32": base.scaled(group_size=3, hash_bits=32, budget=384, prompt_len=800),
    "group_8_b64_protected": base.scaled(group_size=8, budget=300, prompt_len=700, n_sink=4, n_recent=10),
    "group_4_b1": base.scaled(hash_bits=1, budget=200, prompt_len=500),
    "group_1_b2_protected": base.scaled(group_size=1, hash_bits=2, budget=150, prompt_len=600, n_sink=3, n_recent=40),
    "words_6144": base.scaled(n_kv_heads=1, hash_bits=32, budget=6144, prompt_len=6500),
    "bytes_6148": base.scaled(n_kv_heads=1, hash_bits=32, budget=6148, prompt_len=6500, n_sink=4, n_recent=10),
    # one word: the owner table of words wherever it fits a cluster of eight, with and without several units to a CTA
    "words_9984": base.scaled(n_kv_heads=1, hash_bits=32, budget=9984, prompt_len=10300),
    "bytes_9985": base.scaled(n_kv_heads=1, hash_bits=32, budget=9985, prompt_len=10300),
    "words_9472_group_8": base.scaled(n_kv_heads=1, group_size=8, hash_bits=32, budget=9472, prompt_len=9700),
    "bytes_9473_group_8_protected": base.scaled(n_kv_heads=1, group_size=8, hash_bits=32, budget=9473, prompt_len=9700, n_sink=4, n_recent=10),
    "words_10368_group_1": base.scaled(n_kv_heads=1, group_size=1, hash_bits=16, budget=10368, prompt_len=10700),
    "words_9000_over_sms": base.scaled(batch=75, group_size=1, hash_bits=32, head_dim=64, budget=9000, prompt_len=9150),
    "two_words_4096": base.scaled(n_kv_heads=1, budget=4096, prompt_len=4500),
    "two_words_4100": base.scaled(n_kv_heads=1, budget=4100, prompt_len=4500),
    "two_words_6144": base.scaled(n_kv_heads=1, budget=6144, prompt_len=6500),
    "two_words_bytes_6145": base.scaled(n_kv_heads=1, budget=6145, prompt_len=6500),
    "two_words_5632_group_8": base.scaled(n_kv_heads=1, group_size=8, budget=5632, prompt_len=5900),
    "two_words_bytes_5633_group_8_protected": base.scaled(n_kv_heads=1, group_size=8, budget=5633, prompt_len=5900, n_sink=4, n_recent=10),
    # more units than SMs: few-bit codes stay on the CUDA-core kernels, launched plainly behind the hashing
    "few_bits_over_sms": base.scaled(batch=10, n_kv_heads=16, hash_bits=8, group_size=2, budget=400, prompt_len=520, head_dim=64),
    "one_head_groups_over_sms": base.scaled(batch=10, n_kv_heads=16, hash_bits=16, group_size=1, budget=390, prompt_len=520, head_dim=64),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_replay_forms(name):
    case = Case(SHAPES[name])
    case.prefill()
    case.compare_state()
