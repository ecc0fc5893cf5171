"""GPU parity of forwards with fewer work items than SMs, whose items are shared by a cluster of CTAs: parts without key tiles,
two and more parts, tiles of a pair that end in different parts, rows without keys, ragged ends."""
import pytest

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
