"""KVQ_TRACE=1 names the kernels that kvq_drift_metrics launches."""

import os
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parents[1]

SCRIPT = r"""
import torch
from paper_2607_16248_gb300 import kvq
for rows, V in ((2, 50000), (3, 2000), (200, 2000)):
    z = torch.randn(rows, V, device="cuda") * 3
    kvq.drift_metrics(z, z + 0.1, 0.9, 8, 16, 0.02, 0.5)
torch.cuda.synchronize()
"""


def test_drift_trace_lines(kvq_lib):
    env = dict(os.environ, KVQ_TRACE="1", PYTHONPATH=str(ROOT))
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    few, short, many = [l for l in r.stderr.splitlines() if l.startswith("kvq: kvq_drift_metrics ")]
    assert few.endswith("grid (8, 2) x 512")
    assert "grid (3) x 1024, then (8, 3) x 512" in short
    assert "grid (200) x 512, then (8, " in many
