"""GPU parity of the two-stream form (one query tile per CTA): one and two tiles of an item, odd and even numbers of key tiles,
items that begin in either stream, more items than SMs, rows without keys, ragged ends."""
import pytest

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload

from parity_util import compare

pytestmark = pytest.mark.gpu

SHAPES = [
    Workload("two_key_tiles", 1, 2, 2, 256, 256, 64, True, "bf16", 121),
    Workload("odd_walk", 1, 3, 1, 300, 600, 64, False, "fp16", 122),               # 5 key tiles, ragged rows and keys
    Workload("rows_without_keys", 1, 2, 2, 700, 400, 64, True, "fp16", 123),
    Workload("prompt_fp8", 1, 16, 16, 1024, 1024, 128, True, "fp8_e4m3", 124),     # one item per CTA
    Workload("two_rounds", 1, 16, 16, 1500, 1500, 128, True, "bf16", 125, peaked_keys=True),   # 192 items: one or two per CTA
    Workload("three_rounds_full", 3, 12, 2, 1337, 2803, 128, False, "bf16", 126),  # exact mode: 396 items
    Workload("chunk_of_context", 1, 8, 2, 700, 3001, 128, True, "fp8_e4m3", 127),
]


@pytest.fixture(autouse=True)
def _device_status_is_clean():
    binding.device_status_reset()
    yield
    assert binding.device_status() == 0


@pytest.mark.parametrize("mode", [orc.W_EXACT, orc.W_POT, orc.W_H15])
@pytest.mark.parametrize("wl", SHAPES, ids=lambda w: w.name)
def test_two_streams_match_the_oracle(wl, mode):
    rows = None
    if wl.Sq * wl.Sk * wl.Hq * wl.B > 3e7:
        rows = sorted(set(range(0, wl.Sq, 61)) | set(range(max(0, wl.Sq - 130), wl.Sq, 3)) | set(range(0, 130, 3)))
    st = compare(wl, mode, rows=rows, model_p_storage=True)
    assert st["ok"], st


@pytest.mark.parametrize("dtype", ["bf16", "fp8_e4m3"])
@pytest.mark.parametrize("mode", [orc.W_H15K2, orc.W_H15K3])
def test_two_streams_family_members(dtype, mode):
    st = compare(Workload("streams_family", 1, 4, 4, 500, 900, 128, True, dtype, 128), mode, model_p_storage=True)
    assert st["ok"], st
