"""Calls of few rows in the two-kernel form, whose weights are asked of the L2 while the call before still runs, with weights that this call writes:
every step has new ones.  Shares of the contraction that end under the set-up's requests, behind them and beyond all requests, several
row groups."""
import pytest
import torch

import paper_2608_03537_b200 as cf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(40, 2048, 1024), (100, 2304, 2056), (8, 4096, 4096), (33, 2048, 3584), (16, 8192, 4096)])
def test_weights_written_by_the_call_before(M, N, K, cuda_device):
    bf = torch.bfloat16
    g = torch.Generator(device=cuda_device).manual_seed(N + K)
    new = lambda *s: torch.empty(s, device=cuda_device).normal_(generator=g).to(bf)  # noqa: E731
    steps = 6
    X, C, A, zero = [new(N, 64) for _ in range(steps)], new(64, K), new(M, K), torch.zeros(max(N, K), dtype=bf, device=cuda_device)
    weights = torch.zeros(N, K, dtype=bf, device=cuda_device)
    ws = torch.empty(1 << 22, dtype=torch.uint8, device=cuda_device)

    def chain(wait):
        out = torch.full((steps, M, N), float("nan"), dtype=bf, device=cuda_device)
        for i in range(steps):
            cf.gemm_epilogue(X[i], C, weights, cf.EPI_BIAS_RES_LAYERNORM, bias=zero[:K], workspace=ws)
            wait()
            cf.gemm_epilogue(A, weights, out[i], cf.EPI_BIAS_RES_LAYERNORM, bias=zero[:N], workspace=ws, flags=cf.FLAG_B_ROW_MAJOR_NK)
            wait()
        torch.cuda.synchronize()
        return out

    want = chain(torch.cuda.synchronize)
    assert not want.isnan().any() and not torch.equal(want[0], want[1])
    for _ in range(3):
        assert torch.equal(chain(lambda: None), want)
