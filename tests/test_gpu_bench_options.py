"""bench.py as a program: one line that parses, with and without the field solve."""
import json
import os
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("extra", [["--no-field"], ["--learned", "off"]])
def test_bench_prints_one_line(extra, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    detail = tmp_path / "record.json"
    cmd = [sys.executable, "bench.py", "--workload", "1", "--steps", "3", "--warmup", "3", "--also=", "--no-e2e",
           "--no-cpu-baseline", "--fp64-steps", "2", "--adams-steps", "0", "--neumann-steps", "0", "--drift-steps", "0",
           "--min-warmup-s", "0", "--detail", str(detail), *extra]
    r = subprocess.run(cmd, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [x for x in r.stdout.splitlines() if x.strip()]
    assert len(lines) == 1 and len(lines[0]) < 3000
    d = json.loads(lines[0])
    assert d["value"] > 0 and d["status"] == 0 and d["steps"] == 3 and d["gpu_launches"] > 0
    assert ("field_solve" in d) == ("--no-field" not in extra)
    whole = json.loads(detail.read_text())
    assert whole["fp64_mode"]["particle_steps_per_s"] > 0 and (whole["field_solve"] is None) == ("--no-field" in extra)
