"""The benchmark's clock samples with a stand-in for nvidia-smi that takes half a second to start."""
import os
import sys
import time

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = """#!/bin/sh
sleep 0.5
echo "210, 1965, 190.0, Not Active, Not Active, Not Active, Not Active"
while true; do
  sleep 0.02
  echo "1950, 1965, 700.0, Not Active, Not Active, Not Active, Active"
done
"""


def test_a_short_timed_region_is_sampled(tmp_path, monkeypatch):
    sys.path.insert(0, ROOT)
    import bench
    fake = tmp_path / "nvidia-smi"
    fake.write_text(FAKE)
    fake.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    with bench.ClockSampler(0) as clk:
        time.sleep(0.2)
    got = clk.summary()
    assert got["samples"] >= 3 and got["sm_mhz"] == 1950 and got["reasons"] == ["sw_power_cap"], got
