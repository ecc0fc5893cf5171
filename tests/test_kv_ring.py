"""The producer's walk over the K/V ring against a model of its mbarriers (kv_ring_model.cpp): no arrival falls into a phase
that has all of its arrivals, nothing waits for ever, and when the producer gives up its last waits cover every copy."""
import shutil
import subprocess
from pathlib import Path

HERE = Path(__file__).resolve().parent


def test_ring_protocol_holds_for_all_lengths_and_landing_orders(tmp_path):
    exe = tmp_path / "kv_ring_model"
    subprocess.run([shutil.which("g++") or "c++", "-O1", "-std=c++17", "-o", str(exe), str(HERE / "kv_ring_model.cpp")], check=True)
    res = subprocess.run([str(exe), "12"], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr
