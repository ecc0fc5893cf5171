"""Device-free parts of the attention kernels, compiled for the CPU: the producer's walk over the K/V ring against a model of its
mbarriers (kv_ring_model.cpp), and the plans that share work items over CTAs (plan_model.cpp)."""
import shutil
import subprocess
from pathlib import Path

HERE = Path(__file__).resolve().parent


def _run(tmp_path, name, *args):
    exe = tmp_path / name
    subprocess.run([shutil.which("g++") or "c++", "-O1", "-std=c++17", "-o", str(exe), str(HERE / f"{name}.cpp")], check=True)
    res = subprocess.run([str(exe), *args], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr


def test_ring_protocol_holds_for_all_lengths_and_landing_orders(tmp_path):
    """No arrival falls into a phase that has all of its arrivals, nothing waits for ever, and when the producer gives up its last
    waits cover every copy."""
    _run(tmp_path, "kv_ring_model", "12")


def test_plans_follow_the_device(tmp_path):
    _run(tmp_path, "plan_model")


def test_stream_ring_protocol_holds_for_all_lengths_and_landing_orders(tmp_path):
    _run(tmp_path, "stream_ring_model", "12")
