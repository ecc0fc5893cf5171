"""The bounded device-side waits and the sticky status word, exercised without faulting or hanging anything:
a one-warp kernel waits, with a short limit, on a barrier that nothing arrives on; the wait runs out and the
kernel returns with the status word set."""
import numpy as np
import pytest
import torch

from oracle import cpu_oracle as orc
from paper_2609_33586_b200 import binding
from paper_2609_33586_b200.inputs import Workload, make_inputs

from parity_util import compare

pytestmark = pytest.mark.gpu

TIMEOUT = -7      # ATTN_ERR_TIMEOUT
SELFTEST_CODE = (7 << 8) | 0x7F


def test_an_expired_wait_sets_the_sticky_word_and_later_launches_store_nothing_until_reset():
    binding.device_status_reset()
    assert binding.device_status() == 0 and binding.device_status_code() == 0
    try:
        binding.selftest_wait(2_000_000)                       # about a millisecond
        assert binding.device_status() == TIMEOUT
        assert binding.device_status_code() == SELFTEST_CODE
        assert "wait" in binding.status_string(TIMEOUT)

        wl = Workload("after_timeout", 1, 2, 2, 300, 300, 128, True, "bf16", 81)
        inp = make_inputs(wl)
        q, k, v = inp.q.cuda(), inp.k.cuda(), inp.v.cuda()
        out = torch.full((wl.B, wl.Sq, wl.Hq, wl.D), 7.0, dtype=torch.bfloat16, device="cuda")
        lse = torch.full((wl.B, wl.Hq, wl.Sq), -3.0, dtype=torch.float32, device="cuda")
        # the word is sticky: the call itself reports success (it is asynchronous), the kernel stores nothing
        binding.attn_fwd(q, k, v, causal=True, softmax_scale=wl.softmax_scale, weight_mode=orc.W_H15, out=out, lse=lse)
        torch.cuda.synchronize()
        assert torch.all(out == 7.0) and torch.all(lse == -3.0)
        assert binding.device_status() == TIMEOUT and binding.device_status_code() == SELFTEST_CODE   # the first code is kept
        # a second expiry does not replace the first code
        binding.selftest_wait(1_000)
        assert binding.device_status_code() == SELFTEST_CODE
    finally:
        binding.device_status_reset()
    assert binding.device_status() == 0
    # after the reset everything works again
    st = compare(wl, orc.W_H15, inp)
    assert st["ok"], st
    assert binding.device_status() == 0


@pytest.mark.parametrize("wl", [
    Workload("one_key_tile", 1, 2, 2, 300, 100, 128, False, "bf16", 83),
    Workload("rows_without_keys", 1, 2, 2, 300, 20, 64, True, "bf16", 84),
    Workload("several_key_tiles", 1, 2, 2, 600, 600, 128, True, "fp8_e4m3", 85),          # two-stream form
    Workload("several_key_tiles_plain", 4, 40, 8, 300, 500, 128, True, "fp8_e4m3", 88)], ids=lambda w: w.name)
def test_launches_queued_behind_the_expiring_one_store_nothing(wl):
    """No synchronisation in between: the forwards may start (programmatic launch) before the word is set, and warps of one
    block may see it at different times."""
    binding.device_status_reset()
    inp = make_inputs(wl)
    q, k, v = inp.q.cuda(), inp.k.cuda(), inp.v.cuda()
    out = torch.full((wl.B, wl.Sq, wl.Hq, wl.D), 7.0, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((wl.B, wl.Hq, wl.Sq), -3.0, dtype=torch.float32, device="cuda")
    try:
        binding.selftest_wait(200_000)
        for _ in range(8):
            binding.attn_fwd(q, k, v, causal=wl.causal, softmax_scale=wl.softmax_scale, weight_mode=orc.W_H15,
                             q_descale=inp.q_descale, k_descale=inp.k_descale, v_descale=inp.v_descale, out=out, lse=lse)
        torch.cuda.synchronize()
        assert torch.all(out == 7.0) and torch.all(lse == -3.0)
        assert binding.device_status_code() == SELFTEST_CODE
    finally:
        binding.device_status_reset()
    st = compare(wl, orc.W_H15, inp)
    assert st["ok"], st


@pytest.mark.parametrize("wl", [
    Workload("few_rows", 1, 8, 1, 1, 70001, 128, True, "bf16", 86),
    Workload("shared_items", 1, 2, 2, 300, 16384, 128, True, "bf16", 87)], ids=lambda w: w.name)
def test_cluster_kernels_store_nothing_and_do_not_linger_while_the_word_is_set(wl):
    """They take all their steps whatever the word says, and no wait of theirs may last: a few hundred waits one after the
    other, each of which parks for 20 us at most."""
    q = torch.randn(wl.B, wl.Sq, wl.Hq, wl.D, device="cuda").to(torch.bfloat16)
    k = torch.randn(wl.B, wl.Sk, wl.Hkv, wl.D, device="cuda").to(torch.bfloat16)
    kw = dict(causal=True, softmax_scale=wl.softmax_scale, weight_mode=orc.W_H15)
    binding.device_status_reset()
    want, want_lse = binding.attn_fwd(q, k, k, **kw)
    assert binding.device_status() == 0
    out, lse = torch.full_like(want, 7.0), torch.full_like(want_lse, -3.0)
    try:
        binding.selftest_wait(1000)
        assert binding.device_status() == TIMEOUT
        start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        start.record()
        binding.attn_fwd(q, k, k, out=out, lse=lse, **kw)
        end.record()
        torch.cuda.synchronize()
        assert torch.all(out == 7.0) and torch.all(lse == -3.0)
        assert start.elapsed_time(end) < 50.0
    finally:
        binding.device_status_reset()
    binding.attn_fwd(q, k, k, out=out, lse=lse, **kw)
    assert torch.equal(out, want) and torch.equal(lse, want_lse) and binding.device_status() == 0


def test_selftest_limits_are_checked():
    assert binding.lib().attn_selftest_wait(0, None) == -9
    assert binding.lib().attn_selftest_wait(3_000_000_000, None) == -9
    assert binding.device_status() == 0
