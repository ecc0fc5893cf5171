"""GPU parity of forwards with fewer work items than SMs, whose items are shared by a cluster of CTAs: parts without key tiles,
two and more parts, tiles of a pair that end in different parts, rows without keys, ragged ends, and maxima passes whose lengths
lie around the ring's."""
import pytest
import torch

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload, make_inputs

from parity_util import compare

pytestmark = pytest.mark.gpu

SHAPES = [
    Workload("two_parts", 1, 64, 16, 100, 6000, 128, True, "bf16", 101),       # 64 items of one query tile: 2 CTAs each
    Workload("four_parts_fp8", 1, 16, 16, 100, 5000, 128, True, "fp8_e4m3", 102),
    Workload("eight_parts_d64", 1, 2, 2, 300, 4099, 64, False, "fp16", 103),
    Workload("causal_prompt", 1, 1, 1, 3000, 3000, 128, True, "fp8_e4m3", 104, peaked_keys=True),
    Workload("causal_prompt_bf16", 1, 2, 1, 3000, 3000, 64, True, "bf16", 105),
    Workload("few_keys_early", 1, 1, 1, 700, 1900, 128, True, "bf16", 106),
    Workload("fp8_d64", 1, 3, 1, 257, 4500, 64, True, "fp8_e4m3", 107),
]


@pytest.fixture(autouse=True)
def _device_status_is_clean():
    binding.device_status_reset()
    yield
    assert binding.device_status() == 0


IN_DTYPES = {"bf16": binding.IN_BF16, "fp16": binding.IN_FP16, "fp8_e4m3": binding.IN_FP8_E4M3}


def parts_of(wl, mode):
    kernel, ctas = binding.get_plan(wl.B, wl.Hq, wl.Hkv, wl.Sq, wl.Sk, wl.D, wl.causal, mode, IN_DTYPES[wl.in_dtype])
    return ctas if kernel == binding.KERNEL_SHARED else 1


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: w.name)
def test_shared_items_match_the_oracle(wl, mode):
    assert parts_of(wl, mode) > 1 and (wl.name != "two_parts" or parts_of(wl, mode) == 2)
    rows = None
    if wl.Sq * wl.Sk * wl.Hq > 3e7:
        import numpy as np
        rows = np.unique(np.concatenate([np.arange(0, wl.Sq, 17), np.arange(max(0, wl.Sq - 130), wl.Sq)])).astype(np.int32)
    st = compare(wl, mode, rows=rows, model_p_storage=True)
    assert st["ok"], st


def test_two_parts_of_a_pair_of_query_tiles():
    """Planned in the exact mode on 16-bit inputs alone: elsewhere each tile of the pair takes a CTA (two streams)."""
    wl = Workload("two_parts_two_tiles", 1, 48, 12, 200, 6400, 128, True, "bf16", 109)
    assert parts_of(wl, orc.W_EXACT) == 2
    st = compare(wl, orc.W_EXACT, rows=list(range(0, 200, 7)) + [127, 128, 199])
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


# Key tiles, CTAs and the length of the maxima pass that some of them have.  The ring holds 4 tiles at 16 bits and D = 128,
# 8 otherwise; after a pass of odd length one of its positions stays empty.
PASSES = [
    (Workload("pass_3", 1, 2, 2, 256, 3200, 128, False, "bf16", 111), 3),
    (Workload("pass_5", 1, 2, 1, 200, 5200, 128, True, "fp16", 112), 5),
    (Workload("pass_7_two_parts", 1, 48, 48, 100, 3500, 128, True, "bf16", 113), 7),
    (Workload("pass_7_d64", 1, 2, 2, 256, 7200, 64, False, "bf16", 114), 7),
    (Workload("pass_7_fp8", 1, 2, 2, 256, 7200, 128, False, "fp8_e4m3", 115), 7),
    (Workload("pass_9_fp8", 1, 24, 24, 100, 6000, 128, True, "fp8_e4m3", 116), 9),
    (Workload("pass_9_fp8_d64", 2, 16, 16, 80, 4600, 64, False, "fp8_e4m3", 117), 9),
    (Workload("pass_15_fp8_two_parts", 1, 48, 48, 100, 7900, 128, True, "fp8_e4m3", 118), 15),
]


def pass_lengths(tiles, parts):
    """Key tiles that each CTA of a shared item goes over for the row maxima."""
    if parts == 2:
        half = tiles // 2
        return {half // 2, half - half // 2}
    return {(r + 1) * tiles // parts - r * tiles // parts for r in range(parts - 1)}


@pytest.mark.parametrize("mode", [orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl,length", PASSES, ids=lambda x: getattr(x, "name", None))
def test_maxima_passes_around_the_length_of_the_ring(wl, length, mode):
    parts = parts_of(wl, mode)
    assert parts > 1 and length in pass_lengths((wl.Sk + 127) // 128, parts), parts
    inp = make_inputs(wl)
    rows = list(range(0, wl.Sq, 9)) + [wl.Sq - 1]
    st = compare(wl, mode, inp, rows=rows, model_p_storage=True)
    assert st["ok"], st
    # in a stream of calls, where copies land at other times, the result is the same to the bit
    q, k, v = inp.q.cuda(), inp.k.cuda(), inp.v.cuda()
    kw = dict(causal=wl.causal, softmax_scale=wl.softmax_scale, weight_mode=mode, q_descale=inp.q_descale, k_descale=inp.k_descale,
              v_descale=inp.v_descale)
    o, lse = binding.attn_fwd(q, k, v, **kw)
    for _ in range(300):
        again, lse_again = binding.attn_fwd(q, k, v, **kw)
    assert torch.equal(o, again) and torch.equal(lse, lse_again)
