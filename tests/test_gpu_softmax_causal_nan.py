"""Softmax under the causal mask with NaN among the scores: a row is NaN in its live columns where a live score is, and as it would be
without it where the NaN stands above the diagonal, in the row kernel (NaN in each chunk, in the column groups that cross the diagonal and in
those behind it), the cluster kernel and the form for few rows."""
import pytest
import torch

import paper_2608_03537_b200 as cf
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,N,softcap", [(80, 200, 0.0), (80, 504, 0.0), (50, 512, 2.0), (40, 776, 0.0), (24, 1288, 0.0), (8, 1000, 0.0), (2, 64, 0.0), (2, 504, 0.0)])
def test_causal_rows_with_a_nan(batch, N, softcap, cuda_device):
    bf, K = torch.bfloat16, 64
    g = torch.Generator(device=cuda_device).manual_seed(N)
    A, B = (torch.empty(s, device=cuda_device).normal_(generator=g).to(bf) for s in ((batch, N, K), (batch, K, N)))
    A[:, 5, 3] = float("nan")                     # every score of row 5
    column = [(37 * b + 11) % N for b in range(batch)]
    column[1] = N - 1                             # the last row's diagonal alone
    for b in range(1, batch):
        B[b, 7, column[b]] = float("nan")         # from row column[b] on a live one
    Y = torch.zeros(batch, N, N, dtype=bf, device=cuda_device)
    cf.gemm_epilogue(A, B, Y, cf.EPI_SCALE_MASK_SOFTMAX, alpha=K ** -0.5, mask=cf.MASK_CAUSAL, softcap=softcap)
    i, j = torch.arange(N, device=cuda_device)[:, None], torch.arange(N, device=cuda_device)[None, :]
    T = K ** -0.5 * (A.double() @ B.double())
    T = softcap * torch.tanh(T / softcap) if softcap > 0 else T
    want = torch.softmax(T.masked_fill(j > i, float("-inf")), dim=-1)
    live, nan = j <= i, want.isnan().any(dim=-1)
    assert nan[1:, 5].all() and nan[1, N - 1] and not nan[1, 6:N - 1].any()
    assert Y[nan].isnan()[live.expand_as(Y)[nan]].all()
    assert (Y[~nan].double() - want[~nan]).abs().max().item() <= P.TOL_SOFTMAX_MAX
