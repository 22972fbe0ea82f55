"""Row softmax without a mask tensor: one to five 256-column chunks a row, of which the last two are exponentiated once (the last one from
registers, the one before it from its accumulator slot) and the others twice; row ends inside a warp's 32 columns, at and behind
chunk borders, the causal diagonal in the last chunk; scales of both signs and a soft-cap, whose scores are transformed
first; more tiles than CTA pairs, so that the slot order runs across tiles."""
import pytest

import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,M,N,K,causal,softcap,sign", [
    (160, 130, 64, 64, False, 0.0, 1), (80, 256, 256, 64, True, 0.0, 1), (90, 257, 264, 72, False, 0.0, -1), (50, 300, 300 // 8 * 8, 64, False, 2.0, 1),
    (80, 200, 200, 64, True, 0.0, 1), (80, 504, 504, 32, True, 0.0, 1), (40, 512, 512, 64, True, 3.0, 1), (75, 140, 520, 128, False, 0.0, 1),
    (40, 776, 776, 64, True, 0.0, -1), (40, 270, 1000, 64, False, 0.0, 1), (80, 60, 1032, 200, False, 2.0, 1), (20, 1288, 1288, 64, True, 0.0, 1)])
def test_kept_chunks(batch, M, N, K, causal, softcap, sign, cuda_device):
    w = wl.scaled_masked_softmax(batch, M, N, K, seed=M + N, causal=causal, softcap=softcap)
    w.scalars["alpha"] *= sign
    got = P.run_gpu(w, P.dev_tensors(w), fused=True)
    P.check_outputs(w, got, P.run_oracle(w), label=w.name, softmax_tol=P.TOL_SOFTMAX_MAX)
