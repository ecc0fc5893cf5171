"""GPU parity of forwards with fewer work items than SMs, whose items are shared by a cluster of CTAs: parts without key tiles,
two and more parts, tiles of a pair that end in different parts, rows without keys, ragged ends."""
import pytest
import torch

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload

from parity_util import compare

pytestmark = pytest.mark.gpu

SHAPES = [
    Workload("two_parts_chunk", 1, 32, 16, 512, 6000, 128, True, "bf16", 101),       # 64 items: 2 CTAs each
    Workload("four_parts_fp8", 1, 16, 16, 100, 5000, 128, True, "fp8_e4m3", 102),
    Workload("eight_parts_d64", 1, 2, 2, 300, 4099, 64, False, "fp16", 103),
    Workload("causal_prompt", 1, 2, 2, 3000, 3000, 128, True, "fp8_e4m3", 104, peaked_keys=True),
    Workload("causal_prompt_bf16", 1, 4, 2, 2304, 2304, 64, True, "bf16", 105),
    Workload("few_keys_early", 1, 1, 1, 700, 1900, 128, True, "bf16", 106),
    Workload("fp8_d64", 1, 3, 1, 257, 4500, 64, True, "fp8_e4m3", 107),
]


@pytest.fixture(autouse=True)
def _device_status_is_clean():
    binding.device_status_reset()
    yield
    assert binding.device_status() == 0


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: w.name)
def test_shared_items_match_the_oracle(wl, mode):
    rows = None
    if wl.Sq * wl.Sk * wl.Hq > 3e7:
        import numpy as np
        rows = np.unique(np.concatenate([np.arange(0, wl.Sq, 17), np.arange(max(0, wl.Sq - 130), wl.Sq)])).astype(np.int32)
    st = compare(wl, mode, rows=rows, model_p_storage=True)
    assert st["ok"], st


@pytest.mark.parametrize("mode", [orc.W_H15K2, orc.W_H15K3])
def test_shared_items_family_members(mode):
    st = compare(Workload("split_family", 1, 4, 4, 200, 3333, 128, True, "fp8_e4m3", 108), mode, model_p_storage=True)
    assert st["ok"], st


NOT_A_NUMBER = [("bf16", torch.bfloat16), ("fp16", torch.float16), ("fp8_e4m3", torch.float8_e4m3fn)]


@pytest.mark.parametrize("key", [100, 4000, 8190])
@pytest.mark.parametrize("dtype", [d for _, d in NOT_A_NUMBER], ids=[n for n, _ in NOT_A_NUMBER])
def test_a_score_that_is_no_number_shows_in_its_rows(dtype, key):
    """Exact mode, whichever part of the item the key is in: the rows' O is NaN and their LSE -inf, as in the plain form."""
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn(1, s, 2, 64, device="cuda", generator=g) for s in (300, 8192, 8192))
    k[0, key, 0, 3] = float("nan")
    o, lse = binding.attn_fwd(q.to(dtype), k.to(dtype), v.to(dtype), causal=False, softmax_scale=0.125, weight_mode=orc.W_EXACT)
    assert torch.isnan(o[0, :, 0]).all() and torch.isneginf(lse[0, 0]).all()
    assert torch.isfinite(o[0, :, 1]).all() and torch.isfinite(lse[0, 1]).all()


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_that_is_not_finite_shows_even_where_its_part_weighs_nothing(mode, bad):
    """The last key's score lies 700 octaves above all others, so the parts before it weigh 0: 0 times the value is NaN."""
    q = torch.ones(1, 300, 2, 64, device="cuda")
    k = torch.zeros(1, 8192, 2, 64, device="cuda")
    v = torch.ones(1, 8192, 2, 64, device="cuda")
    k[0, 8191] = 64.0
    v[0, 100, 0, 5] = bad
    q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
    o, lse = binding.attn_fwd(q, k, v, causal=False, softmax_scale=0.125, weight_mode=mode)
    assert torch.isnan(o[0, :, 0, 5]).all() and torch.isfinite(lse).all()
    o[0, :, 0, 5] = 0.0
    assert torch.isfinite(o).all()
