"""Softmax behind a short contraction on both sides of the line between the cluster kernel and the row kernel (a whole number of rounds of the
clusters that fit: 33 of 4 CTAs, 7 of 12 and more on a 148-SM device), with and without a mask tensor and a soft-cap."""
import numpy as np
import pytest

import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,N,additive,softcap", [(33, 1024, False, 0.0), (34, 1024, False, 0.0), (33, 768, True, 0.0), (34, 768, True, 0.0), (21, 3064, True, 0.0),
                                                      (22, 3064, True, 0.0), (28, 1792, False, 3.0), (29, 1792, False, 3.0)])
def test_both_sides(batch, N, additive, softcap, cuda_device):
    w = wl.scaled_masked_softmax(batch, 130, N, 64, seed=batch, causal=False, softcap=softcap)
    if additive:
        mask = np.random.default_rng(N).standard_normal((130, N)).astype(np.float32)
        mask[:, ::7] = -np.inf
        w.tensors["mask"] = wl.f32_to_bf16_bits(mask)
    got = P.run_gpu(w, P.dev_tensors(w), fused=True)
    batches = [0, batch // 2, batch - 1]
    P.check_outputs(w, got, P.run_oracle(w, batches=batches), batches=batches, label=w.name)
