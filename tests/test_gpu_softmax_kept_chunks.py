"""Row softmax without a mask tensor: one to five 256-column chunks a row, of which the last two are exponentiated once (the last one from
registers, the one before it from its accumulator slot) and the others twice; row ends inside a warp's 32 columns, at and behind
chunk borders, the causal diagonal in the last chunk; scales of both signs and a soft-cap, whose scores are transformed
first; more tiles than CTA pairs, so that the slot order runs across tiles."""
import pytest
import torch

import paper_2608_03537_b200 as cf
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


@pytest.mark.parametrize("batch,M,N,K", [(80, 200, 64, 64), (80, 250, 504, 64), (60, 30, 776, 64), (40, 300, 1288, 64), (24, 256, 1536, 64)])
def test_rows_with_a_nan_are_nan(batch, M, N, K, cuda_device):
    bf = torch.bfloat16
    g = torch.Generator(device=cuda_device).manual_seed(N)
    A, B = (torch.empty(s, device=cuda_device).normal_(generator=g).to(bf) for s in ((batch, M, K), (batch, K, N)))
    A[:, 1, 3] = float("nan")                            # every score of row 1
    B[3, 5, 6] = float("nan")                            # one score of every row of batch 3
    mask = torch.zeros(M, N, dtype=bf, device=cuda_device)
    mask[2] = float("-inf")                              # a row without a live column is all zero (but in batch 3)
    mask[3, : N - 8] = float("-inf")
    mask[3, N - 3] = float("nan")
    for r in range(4, M - 1, 2):                         # every other row: one score, another column in each
        mask[r, 5 * r % N] = float("nan" if r % 4 else "inf")
    for m in (None, mask):
        Y = torch.zeros(batch, M, N, dtype=bf, device=cuda_device)
        cf.gemm_epilogue(A, B, Y, cf.EPI_SCALE_MASK_SOFTMAX, alpha=K ** -0.5, mask=cf.MASK_NONE if m is None else cf.MASK_ADDITIVE, mask_tensor=m)
        want = torch.zeros(batch, M, 1, dtype=torch.bool, device=cuda_device)
        want[:, 1], want[3] = True, True
        if m is not None:
            want[:, 3], want[:, 4 : M - 1 : 2] = True, True
            assert (Y[:3, 2] == 0).all()
        assert torch.equal(Y.isnan(), want.expand_as(Y))
