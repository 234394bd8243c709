"""The autotuner's file holds measurements of kernels: lines of earlier ones
decide nothing, lines of these are read back by a later process."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _choice(path, measure):
    """rsa_tune in a process of its own, which reads the file afresh."""
    code = ("import json; from paper_1810_06800_gb300 import rsa; "
            f"print(json.dumps(rsa.rsa_tune(64, 4, 100, measure={measure})))")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True,
                       timeout=120, env=dict(os.environ, RSA_TUNE_CACHE=str(path)), check=True)
    return json.loads(r.stdout)


def test_lines_of_earlier_kernels_do_not_count(tmp_path):
    path = tmp_path / "tune.jsonl"
    default = _choice(path, False)
    measured = _choice(path, True)
    again = _choice(path, False)
    for key in ("mode", "threads", "rounds_per_check"):
        assert again[key] == measured[key]
    other = dict(json.loads(path.read_text()), mode="global", threads=0, rounds_per_check=7)
    for kernels in ({}, {"kernels": 1}):
        old = {k: v for k, v in other.items() if k != "kernels"} | kernels
        path.write_text(json.dumps(old) + "\n")
        assert _choice(path, False) == default
    path.write_text(json.dumps(other) + "\n")
    assert _choice(path, False)["rounds_per_check"] == 7
