"""Attention form for short sources and few queries, blocks of 128 source positions and tiles of 128 query rows: one block, full and
partial, under one and two tiles per work item (the second one missing, partial or full); one tile over two to four blocks with
a partial last one; fewer and more work items than SMs, both key layouts; scores that grow from block to block, so that a row's
running maximum is raised (and its output rescaled) after every block, and ones that never raise it.  (3, 129, 136) lies
just across the line to the CTA-pair form."""
import numpy as np
import pytest
import torch

import paper_2608_03537_b200 as cf
import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("growth", [0.0, 3.0, -3.0])
@pytest.mark.parametrize("row_major", [False, True])
@pytest.mark.parametrize("batch,M,S", [(1, 1, 8), (2, 128, 128), (3, 129, 136), (80, 17, 256), (200, 40, 264), (90, 300, 72), (200, 100, 512), (160, 130, 128)])
def test_attention_blocks(batch, M, S, row_major, growth, cuda_device):
    w = wl.target_attention(batch, M, S, 128, seed=batch + M + S)
    w.scalars["alpha"] = 0.12
    # keys scaled up (or down) towards the end of the source: late blocks hold the maxima (or none of them); the factors are powers
    # of two, so that the scaled keys are exact
    K = wl.bf16_to_f64(w.tensors["W1"]) * np.exp2(np.floor(growth * np.arange(S) / S))[None, None, :]
    w.tensors["W1"] = wl.f32_to_bf16_bits(K.astype(np.float32))
    T = P.dev_tensors(w)
    keys = T["W1"].mT.contiguous() if row_major else T["W1"]
    O = P.guarded((batch, M, 128), torch.bfloat16, float("nan"), T["X"].device)
    for _ in range(2):
        cf.b2b_attention(T["X"], keys, T["W2"], O, alpha=w.scalars["alpha"], keys_row_major=row_major)
    torch.cuda.synchronize()
    P.check_outputs(w, {"Y": O}, P.run_oracle(w), label=f"{w.name} growth {growth} row major {row_major}")
