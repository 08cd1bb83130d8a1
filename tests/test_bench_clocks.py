"""The benchmark's record of the clocks in its timed region, with a stand-in for nvidia-smi."""
import os
import stat
import time

import pytest


@pytest.fixture()
def smi(tmp_path, monkeypatch):
    """a program of that name: sleeps, then prints the line in a file every 5 ms"""
    line = tmp_path / "line"

    def make(delay, text, code="while True: print(open(%r).read(), flush=True); time.sleep(0.005)"):
        line.write_text(text)
        exe = tmp_path / "nvidia-smi"
        exe.write_text("#!/usr/bin/env python3\nimport sys, time\ntime.sleep(%r)\n" % delay + (code % str(line) if "%" in code else code) + "\n")
        exe.chmod(exe.stat().st_mode | stat.S_IXUSR)
        monkeypatch.setenv("PATH", str(tmp_path) + os.pathsep + os.environ["PATH"])
        return line

    return make


def test_a_region_shorter_than_the_start_of_nvidia_smi_has_a_record(smi):
    import bench
    line = smi(0.5, "210, 1965, Not Active, Not Active, Not Active, Not Active")
    sampler = bench.ClockSampler(0)
    sampler.start()
    tmp = line.with_suffix(".new")
    tmp.write_text("1935, 1965, Not Active, Not Active, Not Active, Active")
    tmp.rename(line)
    time.sleep(0.2)                                          # (rows of before still on their way)
    sampler.mark()
    record = sampler.stop()
    assert record["samples"] >= 1 and "note" not in record
    assert (record["sm_mhz"], record["sm_max_mhz"], record["reasons"]) == (1935.0, 1965.0, ["sw_power_cap"])


@pytest.mark.parametrize("code,what", [("time.sleep(60)", "no sample in time"), ("sys.exit(9)", "status 9"), ("print('N/A', flush=True); time.sleep(60)", "no sample in time")])
def test_a_record_without_samples_says_why(smi, code, what):
    import bench
    smi(0.0, "", code)
    sampler = bench.ClockSampler(0, patience=0.5)
    sampler.start()
    sampler.mark()
    record = sampler.stop()
    assert record["sm_mhz"] is None and what in record["note"]


def test_a_machine_without_nvidia_smi_says_so(tmp_path, monkeypatch):
    import bench
    monkeypatch.setenv("PATH", str(tmp_path))
    sampler = bench.ClockSampler(0)
    sampler.start()
    sampler.mark()
    assert "nvidia-smi unavailable" in sampler.stop()["note"]
