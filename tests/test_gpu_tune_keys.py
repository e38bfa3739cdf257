"""A tuner's file written when the elimination's variants were others ("inverse/..." 0 to 4, "schur/..." 2 to 4
CTAs a system) chooses nothing now: its lines are kept, and the shapes are tuned under keys of their own."""
import os
import subprocess
import sys

import pytest

from gpu_util import require_lib

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r"""
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_1301_1247_gb300 import hbs
a = torch.eye(300, device="cuda", dtype=torch.complex128).repeat(4, 1, 1)
for _ in range(4):
    assert hbs.batched_inverse(a, 300, 4, 1) == 0
"""


def test_old_choices_are_not_taken_for_cluster_sizes(tmp_path):
    require_lib()
    tune = tmp_path / "tune.txt"
    tune.write_text("inverse/n512/j4/df 0 1.0\n")
    env = dict(os.environ, HBS_AUTOTUNE="1", HBS_TUNE_FILE=str(tune))
    subprocess.run([sys.executable, "-c", CODE, ROOT], check=True, env=env, timeout=300)
    keys = {line.split()[0]: float(line.split()[2]) for line in tune.read_text().splitlines()}
    assert keys["inverse/cluster/n512/j4/df"] > 0 and keys["inverse/n512/j4/df"] < 0
