"""he_attend where no tensor map of the cache can be had (HE_DISABLE_TMA stands for a driver without the encoder): the generic
kernel serves the call, so the outputs are its outputs bit for bit, and differ from the tensor-core kernel's only in rounding."""
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SCRIPT = r"""
import sys, torch
sys.path.insert(0, %r)
from paper_2412_16187_b200 import HashEvictCache
outs = []
for dim, batch, heads, group, budget in ((128, 2, 4, 4, 700), (64, 1, 2, 3, 90)):
    g = torch.Generator(device="cuda").manual_seed(dim)
    c = HashEvictCache(batch, heads, group, dim, 32, [budget] * batch, torch.randn(dim, 32))
    c.k_cache.copy_(torch.randn(c.k_cache.shape, device="cuda", generator=g))
    c.v_cache.copy_(torch.randn(c.v_cache.shape, device="cuda", generator=g))
    c.fill.fill_(budget - 5)
    outs.append(c.attend(torch.randn(batch, heads * group, dim, device="cuda", generator=g).to(torch.bfloat16)).cpu())
torch.save(outs, sys.argv[1])
""" % (ROOT,)


def outputs(path, **env):
    e = {k: v for k, v in os.environ.items() if k not in ("HE_DISABLE_TMA", "HE_DISABLE_ATTEND_MMA")}
    r = subprocess.run([sys.executable, "-c", SCRIPT, str(path)], env=dict(e, **env), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]
    return torch.load(path)


def test_attention_without_tensor_maps_takes_the_generic_kernel(tmp_path):
    default, generic = outputs(tmp_path / "a"), outputs(tmp_path / "b", HE_DISABLE_ATTEND_MMA="1")
    no_map = outputs(tmp_path / "c", HE_DISABLE_TMA="1")
    for x, y, z in zip(default, generic, no_map):
        assert torch.equal(y, z)
        assert not torch.equal(x, y)
        torch.testing.assert_close(x, y, rtol=0, atol=2e-5 * 5)  # 2e-5 of max|V|, as for the oracle
