"""Environment switches that ask something of the tile kernels take effect on calls of few rows too.  They are read once per process, so
each runs in a child; COMFUSE_VERBOSE names every tile kernel when it is first launched."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import workloads as wl
from tests import parity as P
for w in (wl.post_norm(M=40, N=1024, K=264, seed=7, affine=True), wl.scaled_masked_softmax(batch=2, M=512, N=512, K=320, seed=9)):
    P.check_outputs(w, P.run_gpu(w, P.dev_tensors(w)), P.run_oracle(w), label=w.name)
"""


def _launched(**env):
    clean = {k: v for k, v in os.environ.items() if not k.startswith("COMFUSE_")}
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(clean, COMFUSE_VERBOSE="1", PYTHONPATH=ROOT, **env), capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return [line for line in r.stderr.splitlines() if line.startswith("comfuse: kernel")]


def test_switches_reach_calls_of_few_rows(cuda_device):
    assert _launched() == []                                                    # both calls take the form for few rows
    two = _launched(COMFUSE_SOFTMAX_STAGES="2")
    assert len(two) == 1 and "stages=2 lock=0" in two[0], two
    stages = _launched(COMFUSE_SOFTMAX_STAGES="3")
    assert len(stages) == 1 and "stages=3 lock=1" in stages[0], stages
    assert len(_launched(COMFUSE_FEW_ROWS="0")) == 2
    assert len(_launched(COMFUSE_SOFTMAX_CLUSTER="1")) == 1 and len(_launched(COMFUSE_SPLIT_BLOCK="0")) == 1
