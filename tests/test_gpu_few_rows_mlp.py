"""GELU + LayerNorm MLP of few rows (the hidden layer side by side in a cluster), at the edges of its cuts: one row, full and partial
row groups, hidden widths that end inside, at and behind a CTA's 128 units, one to sixteen CTAs, row slices that end empty, both sides of the lines
for narrow hidden layers; without
biases and affine parameters.  Against the fp64 oracle with the bounds of the row-tiled form."""
import pytest
import torch

import paper_2608_03537_b200 as cf
import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("affine", [False, True])
@pytest.mark.parametrize("M,N1", [(1, 8), (3, 1000), (16, 128), (17, 136), (32, 512), (33, 2048), (64, 1920), (65, 384), (300, 520), (900, 256),
                                  (2368, 8), (2369, 8), (3136, 24), (3137, 24), (4736, 40), (4737, 40)])
def test_few_rows_mlp(M, N1, affine, cuda_device):
    w = wl.b2b_mlp(M=M, K=128, N1=N1, N2=128, seed=M + N1, affine=affine)
    P.check_outputs(w, P.run_gpu(w, P.dev_tensors(w), fused=True), P.run_oracle(w), label=w.name)


def test_without_biases(cuda_device):
    w = wl.b2b_mlp(M=50, K=128, N1=400, N2=128, seed=3, affine=False)
    T = P.dev_tensors(w)
    zero = {k: torch.zeros_like(T[k]) for k in ("b1", "b2")}
    O = [torch.full((50, 128), float("nan"), dtype=torch.bfloat16, device=T["X"].device) for _ in range(2)]
    cf.b2b_gemm(T["X"], T["W1"], None, T["W2"], None, O[0], eps=w.scalars["eps"])
    cf.b2b_gemm(T["X"], T["W1"], zero["b1"], T["W2"], zero["b2"], O[1], eps=w.scalars["eps"])
    assert torch.equal(O[0].view(torch.int16), O[1].view(torch.int16)) and bool(torch.isfinite(O[0]).all())
