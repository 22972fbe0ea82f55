"""Masked row softmax: no column's exponentials are worse than the ex2 instruction's, whichever unit they come from (the FMA pipe takes some of
the column pairs).  A relative error e moves a value with mantissa m across a rounding boundary of bf16 with probability 2^7 m e, on
average 185 e, so the share of results that are not the bf16 value nearest to the 64-bit result measures e.  The limit,
1.5e-4, is a mean error of 8e-7: the scores' own rounding and the instruction's 2.4e-7 come to about 0.5e-4."""
import numpy as np
import pytest
import torch

import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,M,N", [(96, 504, 504), (24, 600, 1288), (150, 31, 1288)])
def test_masked_results_are_rounded_once(batch, M, N, cuda_device):
    w = wl.scaled_masked_softmax(batch, M, N, 64, seed=N, causal=False)
    mask = np.random.default_rng(M).standard_normal((M, N)).astype(np.float32)
    mask[:, N - N // 10:] = -np.inf
    w.tensors["mask"] = wl.f32_to_bf16_bits(mask)
    T = P.dev_tensors(w)
    got = P.run_gpu(w, T, fused=True)["Y"]
    want = torch.softmax(w.scalars["alpha"] * (T["A"].double() @ T["B"].double()) + T["mask"].double(), dim=-1)
    wrong = (got != want.to(torch.bfloat16)).double().sum(dim=(0, 1))
    for pair in range(16):  # of each 32 columns
        cols = torch.tensor([c for c in range(N - N // 10) if c // 2 % 16 == pair], device=got.device)
        assert wrong[cols].sum().item() / (batch * M * len(cols)) < 1.5e-4, pair
