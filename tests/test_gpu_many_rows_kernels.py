"""The kernels that calls of many rows take, at the small and ragged sizes of the suite.  Calls of few rows have a form of their own, which
takes nearly every size that is small enough for the oracle; here the same tests run once more in a child process in which that
form is off (COMFUSE_FEW_ROWS=0), and the softmax ones in one in which the cluster kernel is forced.  The switches are read
once per process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FEW_ROWS_OFF, CLUSTER = {"COMFUSE_FEW_ROWS": "0"}, {"COMFUSE_SOFTMAX_CLUSTER": "1"}


@pytest.mark.parametrize("files,select,env", [
    (["test_gpu_gemm_epilogue.py", "test_gpu_softmax_mask_boxes.py"], "", FEW_ROWS_OFF),
    (["test_gpu_random_shapes.py"], "", FEW_ROWS_OFF),
    (["test_gpu_b2b.py", "test_gpu_host_io.py", "test_gpu_back_to_back.py"], "", FEW_ROWS_OFF),
    (["test_gpu_gemm_epilogue.py", "test_gpu_random_shapes.py"], "softmax or test_random_shape_and_operands", CLUSTER),
], ids=["gemm", "random", "b2b", "softmax-cluster"])
def test_suite_with_the_form_for_few_rows_off(files, select, env, cuda_device):
    assert "COMFUSE_FEW_ROWS" not in os.environ and "COMFUSE_SOFTMAX_CLUSTER" not in os.environ
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-m", "gpu", "-p", "no:cacheprovider", *(["-k", select] if select else []), *(os.path.join("tests", f) for f in files)]
    r = subprocess.run(cmd, cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT, **env), capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-4000:] + r.stderr[-2000:]
