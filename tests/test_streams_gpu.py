"""GPU parity of the two-stream form (one query tile per CTA): one and two tiles of an item, odd and even numbers of key tiles,
items that begin in either stream, more items than SMs, rows without keys, ragged ends."""
import pytest
import torch

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload, make_inputs

from parity_util import PLAIN, STREAMS, compare, plan_of

pytestmark = pytest.mark.gpu

SHAPES = [
    Workload("two_key_tiles", 1, 2, 2, 256, 256, 64, True, "bf16", 121),
    Workload("odd_walk", 1, 3, 1, 300, 600, 64, False, "fp16", 122),               # 5 key tiles, ragged rows and keys
    Workload("rows_without_keys", 1, 2, 2, 700, 400, 64, True, "fp16", 123),
    Workload("prompt_fp8", 1, 16, 16, 1024, 1024, 128, True, "fp8_e4m3", 124),     # one item per CTA
    Workload("two_rounds", 1, 16, 16, 1500, 1500, 128, True, "bf16", 125, peaked_keys=True),   # 192 items: one or two per CTA
    Workload("chunk_of_context", 1, 20, 4, 700, 2000, 128, True, "fp8_e4m3", 127),
    # more items than SMs, with two staged query tiles and four pairs of ring slots
    Workload("two_rounds_fp8", 1, 16, 16, 1664, 1664, 128, True, "fp8_e4m3", 133),       # 13 key tiles
    Workload("two_rounds_d64", 1, 16, 16, 1664, 1664, 64, True, "bf16", 134, peaked_keys=True),
    Workload("two_rounds_full", 4, 64, 8, 100, 1100, 128, False, "fp8_e4m3", 135),       # 256 items of 9 key tiles
]
THREE_ROUNDS = Workload("three_rounds_full", 3, 12, 2, 1337, 2803, 128, False, "bf16", 126)


@pytest.fixture(autouse=True)
def _device_status_is_clean():
    binding.device_status_reset()
    yield
    assert binding.device_status() == 0


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: w.name)
def test_two_streams_match_the_oracle(wl, mode):
    assert plan_of(wl, mode) == STREAMS
    rows = None
    if wl.Sq * wl.Sk * wl.Hq * wl.B > 3e7:
        rows = sorted((set(range(0, wl.Sq, 61)) | set(range(max(0, wl.Sq - 130), wl.Sq, 3)) | set(range(0, 130, 3))) & set(range(wl.Sq)))
    st = compare(wl, mode, rows=rows, model_p_storage=True)
    assert st["ok"], st


def test_two_streams_over_three_rounds_of_items():
    assert plan_of(THREE_ROUNDS, orc.W_EXACT) == STREAMS      # 396 items; the rounding maps take the plain form
    st = compare(THREE_ROUNDS, orc.W_EXACT, rows=sorted(set(range(0, 1337, 61)) | set(range(1207, 1337, 3)) | set(range(0, 130, 3))))
    assert st["ok"], st


@pytest.mark.parametrize("dtype", ["bf16", "fp8_e4m3"])
@pytest.mark.parametrize("mode", [orc.W_H15K2, orc.W_H15K3])
def test_two_streams_family_members(dtype, mode):
    wl = Workload("streams_family", 1, 4, 4, 500, 900, 128, True, dtype, 128)
    assert plan_of(wl, mode) == STREAMS
    st = compare(wl, mode, model_p_storage=True)
    assert st["ok"], st


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl,copies", [
    (Workload("anchor_full", 1, 12, 2, 1337, 700, 128, False, "bf16", 129), 12),
    (Workload("anchor_causal", 1, 16, 4, 1000, 1000, 128, True, "bf16", 130, peaked_keys=True), 8),
    (Workload("anchor_fp16_d64", 1, 8, 8, 700, 700, 64, True, "fp16", 131), 24),
    (Workload("anchor_fp8", 1, 16, 16, 1000, 1000, 128, True, "fp8_e4m3", 132), 8)], ids=lambda x: getattr(x, "name", None))
def test_two_streams_round_p_as_the_plain_form_does(wl, copies, mode):
    """The same heads, alone (two streams) and among many (plain form): P has the same bits, so that O differs by fp32 sums alone.
    Those move O by less than 2^-16 of itself before it is rounded to bf16, so at most 2 x 2^-16 / 2^-8 of its values fall on the
    other side of a rounding and move by up to 2^-8 (2-norm sqrt(2^-7) 2^-8 = 3.5e-4).  P rounded about the maxima of a stream's own
    tiles moves O by 2e-3 in the exact mode on 16-bit inputs."""
    inp = make_inputs(wl)
    q, k, v = inp.q.cuda(), inp.k.cuda(), inp.v.cuda()
    many = [x.expand(copies, *x.shape[1:]).contiguous() if x.dtype != torch.float8_e4m3fn else
            x.view(torch.uint8).expand(copies, *x.shape[1:]).contiguous().view(x.dtype) for x in (q, k, v)]
    assert plan_of(wl, mode) == STREAMS and plan_of(wl.with_(B=copies), mode) == PLAIN
    kw = dict(causal=wl.causal, softmax_scale=wl.softmax_scale, weight_mode=mode, q_descale=inp.q_descale, k_descale=inp.k_descale,
              v_descale=inp.v_descale)
    o, lse = binding.attn_fwd(q, k, v, **kw)
    want, want_lse = binding.attn_fwd(*many, **kw)
    o, want = o[0].double(), want[copies // 2].double()
    assert ((o - want).norm() / want.norm()).item() < 3.5e-4
    assert (lse[0] - want_lse[copies // 2]).abs().max().item() < 1e-5


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_H15])
@pytest.mark.parametrize("wl", [SHAPES[1], SHAPES[3], SHAPES[6]], ids=lambda w: w.name)
def test_two_streams_give_the_same_bits_in_a_stream_of_calls(wl, mode):
    assert plan_of(wl, mode) == STREAMS
    inp = make_inputs(wl)
    q, k, v = inp.q.cuda(), inp.k.cuda(), inp.v.cuda()
    kw = dict(causal=wl.causal, softmax_scale=wl.softmax_scale, weight_mode=mode, q_descale=inp.q_descale, k_descale=inp.k_descale,
              v_descale=inp.v_descale)
    o, lse = binding.attn_fwd(q, k, v, **kw)
    for _ in range(300):
        again, lse_again = binding.attn_fwd(q, k, v, **kw)
    assert torch.equal(o, again) and torch.equal(lse, lse_again)


@pytest.mark.parametrize("key", [5, 130, 690])       # in the first tile of either stream and in the last tile
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float8_e4m3fn])
def test_two_streams_show_a_score_that_is_no_number(dtype, key):
    """Exact mode: the rows' O is NaN and their LSE -inf, as in the plain form."""
    assert plan_of(Workload("nan", 1, 2, 2, 300, 700, 64, False, {torch.bfloat16: "bf16", torch.float16: "fp16"}.get(dtype, "fp8_e4m3"), 0), orc.W_EXACT) == STREAMS
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn(1, s, 2, 64, device="cuda", generator=g) for s in (300, 700, 700))
    k[0, key, 0, 3] = float("nan")
    o, lse = binding.attn_fwd(q.to(dtype), k.to(dtype), v.to(dtype), causal=False, softmax_scale=0.125, weight_mode=orc.W_EXACT)
    assert torch.isnan(o[0, :, 0]).all() and torch.isneginf(lse[0, 0]).all()
    assert torch.isfinite(o[0, :, 1]).all() and torch.isfinite(lse[0, 1]).all()


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("key", [100, 200])
def test_two_streams_show_a_value_that_is_not_finite_where_its_stream_weighs_nothing(key, bad, mode):
    """The last key's score lies 700 octaves above all others, so everything before it weighs 0: 0 times the value is NaN."""
    assert plan_of(Workload("inf", 1, 2, 2, 300, 700, 64, False, "bf16", 0), mode) == STREAMS
    q = torch.ones(1, 300, 2, 64, device="cuda")
    k = torch.zeros(1, 700, 2, 64, device="cuda")
    v = torch.ones(1, 700, 2, 64, device="cuda")
    k[0, 699] = 64.0
    v[0, key, 0, 5] = bad
    q, k, v = (x.to(torch.bfloat16) for x in (q, k, v))
    o, lse = binding.attn_fwd(q, k, v, causal=False, softmax_scale=0.125, weight_mode=mode)
    assert torch.isnan(o[0, :, 0, 5]).all() and torch.isfinite(lse).all()
    o[0, :, 0, 5] = 0.0
    assert torch.isfinite(o).all()
