"""bench.py's waits have a limit: a device that never finishes ends the run
with the stage's name and what was measured, not after the caller's patience."""

import os
import subprocess
import sys
import time

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


class NeverDone:
    """An event that never completes."""

    def __init__(self, enable_timing=False):
        pass

    def record(self, stream):
        pass

    def query(self):
        return False


class FakeTorch:
    class cuda:
        Event = NeverDone

        @staticmethod
        def synchronize(dev=None):
            raise AssertionError("an unlimited wait on a device that has not finished")


def test_wait_on_an_event_that_never_completes(monkeypatch, capsys):
    import bench
    stages = bench.Stages(limit_s=0.2)
    monkeypatch.setattr(bench, "STAGES", stages)
    stages.start("eager epochs")
    stages.measured["ms"] = 7.5
    t0 = time.monotonic()
    with pytest.raises(bench.StageTimeout) as e:
        bench._timed_loop(FakeTorch, None, lambda: None, 1)
    assert 0.2 <= time.monotonic() - t0 < 5.0
    assert "eager epochs" in str(e.value) and '"ms": 7.5' in str(e.value)
    assert "eager epochs" in capsys.readouterr().err


def test_a_stopped_stage_ends_the_process(tmp_path):
    code = ("import bench\n"
            "bench.STAGES.limit_s = 0.2\n"
            "def run():\n"
            "    bench.STAGES.start('end to end')\n"
            "    bench.STAGES.measured['ms_per_step_graph'] = 7.7\n"
            "    bench.STAGES.wait(lambda: False)\n"
            "bench.guarded(run)\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=60)
    assert r.returncode == 3
    assert r.stdout == "" and "end to end" in r.stderr and "7.7" in r.stderr
