"""The block replay on data whose steps depend on one another: queries that repeat (constant, near-constant, four in turn) and keys
that repeat, so that most of a block is walked through step by step. Against the oracle at the edges of that walk, and its time
against the same shape with independent queries."""
import numpy as np
import pytest
import torch

from cases import C
from paper_2412_16187_b200 import HashEvictCache
from parity import Case, to_dev

pytestmark = pytest.mark.gpu

base = C["throughput_batch"].scaled(batch=1, n_kv_heads=2, ragged=False)
SHAPES = {
    **{f"budget_{c}": base.scaled(budget=c, prompt_len=c + 200) for c in (1, 31, 127, 385, 1537)},
    **{f"group_{g}": base.scaled(group_size=g, hash_bits=b, budget=390, prompt_len=777) for g, b in ((1, 8), (1, 64), (3, 32), (4, 32), (8, 64))},
    "one_step_left": base.scaled(budget=300, prompt_len=300 + 129, hash_bits=32),
    "protected": base.scaled(budget=700, prompt_len=1100, hash_bits=16, n_sink=4, n_recent=10),
    "protected_two_words": base.scaled(budget=1600, prompt_len=2000, n_sink=4, n_recent=10),
    "protected_one_recent": base.scaled(budget=130, prompt_len=400, hash_bits=32, n_sink=0, n_recent=1),
    "protected_sinks_only": base.scaled(budget=130, prompt_len=400, hash_bits=32, group_size=3, n_sink=128, n_recent=0),
    "protected_window_of_a_block": base.scaled(budget=1600, prompt_len=2000, hash_bits=32, n_sink=2, n_recent=127),
    "cluster": base.scaled(n_kv_heads=1, hash_bits=32, budget=4096, prompt_len=4500),
    "cluster_protected": base.scaled(n_kv_heads=1, hash_bits=32, budget=4096, prompt_len=4500, n_sink=4, n_recent=10),
    "blocks_of_64": base.scaled(n_kv_heads=1, budget=8700, prompt_len=8900),
}


def repeat_rows(x, how):
    """x [B, heads, N, d]: the first row(s) of every head in place of all; "near" keeps a tenth of the variation."""
    out = np.empty(x.shape, x.dtype)
    if how in ("constant", "four"):
        out[:] = x[:, :, np.arange(x.shape[2]) % (4 if how == "four" else 1)]
        return out
    f = torch.from_numpy(x.view(np.int16)).view(torch.bfloat16).float()
    out[:] = (f[:, :, :1] + 0.1 * f).to(torch.bfloat16).view(torch.int16).numpy().view(np.uint16)
    return out


@pytest.mark.parametrize("name", list(SHAPES))
def test_repeating_queries(name):
    for how in ("constant", "near", "four"):
        case = Case(SHAPES[name])
        case.Q = repeat_rows(case.Q, how)
        case.dQ = to_dev(case.Q, case.w)
        case.prefill()
        case.compare_state()


@pytest.mark.parametrize("name", ["budget_385", "group_1", "group_3", "protected", "cluster_protected"])
def test_repeating_keys(name):
    for how in ("constant", "four"):
        case = Case(SHAPES[name])
        case.K = repeat_rows(case.K, how)
        case.dK = to_dev(case.K, case.w)
        case.prefill()
        case.compare_state()


def test_constant_queries_cost_a_bounded_multiple():
    """A block of 128 steps settles in about 12 000 cycles here when its steps are independent. Walked step by step, 2048 slots take
    some 400 cycles each, and the passes before that no more than as much again: 8 times. (Evaluated in passes alone: 50 times.)"""
    heads, slots, tokens, dim, bits = 32, 2048, 4096, 128, 32
    g = torch.Generator(device="cuda").manual_seed(3)
    k = torch.randn(1, heads, tokens, dim, device="cuda", generator=g).to(torch.bfloat16)
    q = torch.randn(1, heads, tokens, dim, device="cuda", generator=g).to(torch.bfloat16)
    same = q[:, :, :1].expand_as(q).contiguous()
    c = HashEvictCache(1, heads, 1, dim, bits, [slots], torch.randn(dim, bits))
    length = torch.tensor([tokens], dtype=torch.int32, device="cuda")

    def time(queries):
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            c.prefill_compress(queries, k, k, length)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return sorted(times[1:])[2]

    assert time(same) < 12 * time(q)
