"""The reference arm of bench.py on the CPU: more than one step, on a few small instances. Its first step
keeps the solutions for scoring, the others do not, and it prints one JSON line."""
import argparse
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

from paper_2601_14414_gb300 import workloads as W  # noqa: E402


def test_reference_arm_runs_several_steps(monkeypatch, capsys):
    insts = [W.random_ltv(400 + j, 3, 1, 6) for j in range(6)]
    monkeypatch.setattr(W, "batched_uneven", lambda seed, batch: insts)
    monkeypatch.setattr(bench, "REF_STEP_SECONDS", 0.0)
    for key in ("RANK", "WORLD_SIZE", "LOCAL_RANK"):
        monkeypatch.delenv(key, raising=False)
    assert bench.run_reference(argparse.Namespace(batch=6, warmup=3, steps=3, gpus=1)) == 0
    lines = capsys.readouterr().out.strip().splitlines()
    assert len(lines) == 1
    got = json.loads(lines[0])
    assert got["impl"] == "reference" and got["steps"] == 3 and got["warmup"] == 3 and got["n_gpus"] == 1
    assert got["accuracy"]["of"] == 6 and got["accuracy"]["ok"] == 6
    assert got["value"] > 0 and got["ms_per_step"] > 0 and "unavailable" not in got
