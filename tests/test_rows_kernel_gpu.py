"""GPU parity of forwards with few query rows per key/value head (decoding, short chunks), which run on a kernel of their
own: the edges of its row tiles (16, 32, 64), of its key tiles, of the split over a cluster and of a round of TMEM."""
import pytest
import torch

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload

from parity_util import compare

pytestmark = pytest.mark.gpu

ALL = [orc.W_EXACT, orc.W_POT, orc.W_H15]

SHAPES = [
    # name, B, Hq, Hkv, Sq, Sk, D, causal, dtype
    Workload("one_key", 1, 4, 1, 1, 1, 128, True, "bf16", 81),
    Workload("one_tile", 2, 2, 2, 1, 128, 64, True, "bf16", 82),
    Workload("tile_plus_one", 1, 12, 2, 1, 129, 128, True, "fp16", 83),
    Workload("rows_16", 1, 16, 4, 4, 1000, 128, True, "bf16", 84, peaked_keys=True),
    Workload("rows_17", 1, 1, 1, 17, 777, 64, True, "fp8_e4m3", 85),
    Workload("rows_32_full", 2, 8, 2, 8, 500, 128, False, "fp8_e4m3", 86),
    Workload("rows_33", 1, 3, 1, 11, 901, 128, True, "bf16", 87),
    Workload("rows_64", 1, 32, 8, 16, 1500, 128, True, "fp8_e4m3", 88),
    Workload("rows_without_keys", 1, 2, 1, 20, 9, 64, True, "fp16", 89),
    Workload("many_groups", 10, 32, 32, 2, 300, 64, True, "bf16", 90),   # more (batch, head) pairs than SMs
    Workload("one_tile_many_heads", 32, 32, 8, 3, 100, 64, True, "fp8_e4m3", 96),
    Workload("no_keys_many_heads", 32, 32, 8, 3, 2, 64, True, "bf16", 97),
    Workload("rows_33_of_many", 40, 66, 2, 1, 260, 128, True, "fp16", 98),
    Workload("rounds_n16", 1, 1, 1, 1, 70001, 64, True, "bf16", 91),     # more than 16 x 32 key tiles
    Workload("rounds_n64", 1, 4, 1, 15, 17000, 128, True, "bf16", 92),   # more than 16 x 8
    Workload("rounds_n32_fp8", 1, 8, 1, 4, 40000, 128, True, "fp8_e4m3", 93),
]

# Shapes that the few-row kernel could take, of so few keys that the plain or the two-stream form is faster.
PLAIN = {"one_key", "one_tile", "tile_plus_one", "rows_without_keys"}
STREAMS = {"rows_32_full"}


@pytest.fixture(autouse=True)
def _device_status_is_clean():
    binding.device_status_reset()
    yield
    assert binding.device_status() == 0


@pytest.mark.parametrize("mode", ALL)
@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: w.name)
def test_few_rows_match_the_oracle(wl, mode):
    dt = {"bf16": binding.IN_BF16, "fp16": binding.IN_FP16, "fp8_e4m3": binding.IN_FP8_E4M3}[wl.in_dtype]
    kernel, _ = binding.get_plan(wl.B, wl.Hq, wl.Hkv, wl.Sq, wl.Sk, wl.D, wl.causal, mode, dt)
    assert kernel == (binding.KERNEL_PLAIN if wl.name in PLAIN else binding.KERNEL_STREAMS if wl.name in STREAMS else binding.KERNEL_FEW_ROWS), wl.name
    st = compare(wl, mode, model_p_storage=True)
    assert st["ok"], st


@pytest.mark.parametrize("mode", [orc.W_H15K2, orc.W_H15K3])
@pytest.mark.parametrize("dtype", ["bf16", "fp8_e4m3"])
def test_few_rows_family_members(dtype, mode):
    st = compare(Workload("rows_family", 2, 12, 2, 1, 2100, 128, True, dtype, 94), mode, model_p_storage=True)
    assert st["ok"], st


@pytest.mark.parametrize("dtype", ["bf16", "fp16", "fp8_e4m3"])
def test_few_rows_dropped_tail(dtype):
    st = compare(Workload("rows_drop", 1, 8, 2, 3, 900, 128, True, dtype, 95), orc.W_POT, pot_tail=(8, True),
                 allow_output_rounding=True)
    assert st["ok"], st


def test_few_rows_nothing_is_stored_while_the_status_word_is_set():
    q = torch.randn(1, 1, 8, 128, device="cuda").to(torch.bfloat16)
    k = torch.randn(1, 3000, 2, 128, device="cuda").to(torch.bfloat16)
    out = torch.full((1, 1, 8, 128), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((1, 8, 1), 7.0, device="cuda")
    binding.selftest_wait(1000)
    torch.cuda.synchronize()
    assert binding.device_status() == -7
    binding.attn_fwd(q, k, k, causal=True, softmax_scale=0.1, weight_mode=orc.W_H15, out=out, lse=lse)
    torch.cuda.synchronize()
    assert torch.all(out == 7.0) and torch.all(lse == 7.0)
    binding.device_status_reset()
    binding.attn_fwd(q, k, k, causal=True, softmax_scale=0.1, weight_mode=orc.W_H15, out=out, lse=lse)
    torch.cuda.synchronize()
    assert torch.all(out != 7.0)


@pytest.mark.parametrize("key", [100, 4000, 8190])
@pytest.mark.parametrize("rows", [1, 20, 50])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16, torch.float8_e4m3fn])
def test_few_rows_show_a_score_that_is_no_number(dtype, rows, key):
    g = torch.Generator(device="cuda").manual_seed(6)
    q, k, v = (torch.randn(1, s, 2, 128, device="cuda", generator=g) for s in (rows, 8192, 8192))
    k[0, key, 0, 3] = float("nan")
    o, lse = binding.attn_fwd(q.to(dtype), k.to(dtype), v.to(dtype), causal=False, softmax_scale=0.0625, weight_mode=orc.W_EXACT)
    assert torch.isnan(o[0, :, 0]).all() and torch.isneginf(lse[0, 0]).all()
    assert torch.isfinite(o[0, :, 1]).all() and torch.isfinite(lse[0, 1]).all()
