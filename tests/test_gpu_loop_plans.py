"""The launch shapes of the loop k-sums come from the shape of the model alone: models of one shape sum in the same order, to
the bit, whatever the process has launched before.  Each case starts a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import torch
from paper_1710_08830_gb300 import api, inputs
spec = {spec}
def loops():
    m = api.Model(spec, api.{precision})
    return m.loops(0.1)
first = loops()
assert torch.equal(first, loops())
"""


# more than 48 KB of shared memory (six states FP64; two bands FP64, three y differences, and FP32 with five on a large fine
# mesh), and less
@pytest.mark.parametrize("spec,precision", [
    ("inputs.t2g_soc(0, 0.2, 2.0, 0.4, Lq=8, nc=6, n_ff=9)", "FP64"), ("inputs.t2g_soc(0, 0.2, 2.0, 0.4, Lq=5, nc=5, n_ff=13)", "FP64"),
    ("inputs.rashba_bilayer(Lq=8, nc=5, n_ff=13)", "FP64"), ("inputs.rashba_bilayer(Lq=12, nc=5, n_ff=9)", "SPLIT32"),
    ("inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.818, Lq=13, nc=17, n_ff=9)", "FP64"),
    ("inputs.rashba_hubbard(1.0, -0.2, 0.3, 2.5, -0.818, Lq=7, nc=100, n_ff=13)", "SPLIT32")])
def test_models_of_one_shape_sum_in_one_order(spec, precision):
    r = subprocess.run([sys.executable, "-c", CODE.format(spec=spec, precision=precision)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
