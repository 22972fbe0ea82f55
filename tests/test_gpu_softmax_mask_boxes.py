"""Row softmax with an additive mask whose boxes share the epilogue warps' staging buffers: one to several tiles per CTA pair
(more tiles than pairs, so that a box is refilled across tiles), row lengths that end inside, at and behind a warp's 64
columns and a 256-column chunk, row counts that leave whole boxes outside the mask
(whose warps hand the accumulators back unread); up to a warp of rows of more than 512 columns, whose threads read the mask
themselves."""
import numpy as np
import pytest

import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,M,N,K,softcap", [(1, 1, 64, 8, 0.0), (3, 31, 72, 64, 0.0), (90, 129, 200, 64, 0.0), (160, 33, 256, 64, 3.0), (80, 257, 264, 32, 0.0),
                                                 (40, 130, 520, 128, 0.0), (40, 300, 776, 64, 2.0), (35, 70, 1032, 256, 0.0), (160, 33, 64, 64, 0.0), (160, 31, 72, 64, 0.0), (134, 1, 720, 88, 0.0),
                                                 (150, 20, 304, 16, 0.0), (90, 165, 1176, 104, 2.0), (190, 32, 1056, 64, 2.0),
                                                 (190, 33, 1056, 64, 0.0), (150, 9, 600, 32, 0.0)])
def test_additive_mask_boxes(batch, M, N, K, softcap, cuda_device):
    w = wl.scaled_masked_softmax(batch, M, N, K, seed=M + N, causal=False, softcap=softcap)
    g = np.random.default_rng(N)
    mask = (g.standard_normal((M, N)) * 2.0).astype(np.float32)
    mask[g.random((M, N)) < 0.2] = -np.inf
    mask[M // 2, :] = -np.inf
    w.tensors["mask"] = wl.f32_to_bf16_bits(mask)
    got = P.run_gpu(w, P.dev_tensors(w), fused=True)
    P.check_outputs(w, got, P.run_oracle(w), label=w.name, softmax_tol=P.TOL_SOFTMAX_MAX)
    assert (got["Y"][:, M // 2, :] == 0).all() and (got["Y"][:, mask_of(mask)] == 0).all()


def mask_of(mask):
    import torch
    return torch.from_numpy(np.isneginf(mask))
