"""The C-ABI library loads and exports every symbol that include/attn.h declares (no GPU needed)."""
import ctypes
import os
import re
import subprocess
import sys
from pathlib import Path

import torch

from paper_2609_33586_b200 import binding, build

ROOT = Path(__file__).resolve().parent.parent


def _declared_functions():
    text = (ROOT / "include" / "attn.h").read_text()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(attn_[a-z_0-9]+)\s*\(", text)))


def test_library_builds_and_exports_every_declared_symbol():
    lib_path = build.build()
    L = ctypes.CDLL(str(lib_path))
    declared = _declared_functions()
    assert set(declared) == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(L, name), name


def test_host_only_entry_points_work_without_a_gpu():
    assert binding.version().startswith("rowmax-attn-b200")
    assert binding.status_string(0) == "ok" and "shape" in binding.status_string(-2)
    for in_dtype, mode, fmt, off in ((0, 2, binding.P_BF16, 0), (1, 0, binding.P_E4M3, 8), (1, 2, binding.P_E5M2, 15),
                                     (1, 3, binding.P_E5M2, 15), (1, 4, binding.P_E4M3, 8), (1, 5, binding.P_E4M3, 8)):
        s = binding.get_schedule(128, in_dtype, mode, True)
        assert (s["tile_m"], s["tile_n"], s["kv_order"], s["rescale_tau"], s["pot_kmax"]) == (128, 128, 1, 0.0, 20)
        assert (s["p_format"], s["p_offset_log2"]) == (fmt, off)
    assert binding.lib().attn_get_schedule(96, 0, 0, 0, *([None] * 7)) == -2
    # argument validation happens before any CUDA call
    assert binding.attn_fwd_raw(None, None, None, None, None, 1, 1, 1, 1, 1, 64, 0, 1.0, 0, 0, 1, 1, 1, None) == -1
    assert binding.lib().attn_get_plan(1, 3, 2, 64, 64, 64, 0, 0, 0, None, None) == -2
    assert binding.lib().attn_weight_map(None, None, 0, 2, None) == 0
    assert binding.lib().attn_weight_map(None, None, 4, 2, None) == -1


def test_only_attn_fwd_needs_the_host_module():
    code = """
import sys
sys.modules["paper_2609_33586_b200._host"] = None      # its import fails
from paper_2609_33586_b200 import binding
import torch
assert binding.version() and binding.launch_count() == 0 and binding.get_schedule(64, 0, 0, True)["tile_n"] == 128
x = torch.zeros(1, 1, 1, 64, dtype=torch.bfloat16)
try:
    binding.attn_fwd(x, x, x, causal=True, softmax_scale=1.0, weight_mode=0)
except RuntimeError as e:
    assert "host module" in str(e)
else:
    raise SystemExit("no error")
"""
    subprocess.run([sys.executable, "-c", code], check=True, cwd=ROOT, env=dict(os.environ, PYTHONPATH=str(ROOT)))


def test_a_host_module_built_for_another_torch_is_not_current(tmp_path):
    built = build.build_host()
    assert build.host_is_current(built, torch.__version__)
    assert not build.host_is_current(built, torch.__version__ + "1") and not build.host_is_current(built, torch.__version__[:-1])
    assert not build.host_is_current(tmp_path / "absent.so", torch.__version__)
    binding.host_forward()
