"""Additive masks whose masked entries are finite, from -1e4 to the lowest bf16, in each kernel that takes a mask: masks that leave no live column
to whole 64-column groups (a causal mask, a window and a padding mask given as data) and to whole rows; and a window of scores
far below the others without a mask.

The reference adds score and mask in fp32, as every kernel does, and goes on in 64 bits: a row in which every score is masked with
-1e9 or less has equal sums and so the probabilities 1/N, in 64 bits throughout it would have those of the unmasked scores."""
import numpy as np
import pytest

import workloads as wl
from oracle import comfuse_oracle as orc
from tests import parity as P

pytestmark = pytest.mark.gpu

LOWEST = -3.3895313892515355e38
FILLS = [-1e4, -1e9, -1e10, -1e20, -1e30, -1e38, LOWEST]


def finite_mask(M, N, fill):
    """Rows in turn: causal (of columns scaled to N), a window, padding in front, no live column."""
    i, j = np.arange(M)[:, None], np.arange(N)[None, :]
    at = i * N // M
    live = np.select([i % 4 == 0, i % 4 == 1, i % 4 == 2], [j <= at, np.abs(j - at) <= 20, j >= N // 2], False)
    bias = np.random.default_rng(M + N).standard_normal((M, N))
    return wl.f32_to_bf16_bits(np.where(live, bias, fill).astype(np.float32))


def reference(w):
    T = w.scalars["alpha"] * orc.gemm(wl.bf16_to_f64(w.tensors["A"]), wl.bf16_to_f64(w.tensors["B"]))
    cap = w.scalars["softcap"]
    T = cap * np.tanh(T / cap) if cap > 0 else T
    return {"Y": orc.softmax_rows((T.astype(np.float32) + wl.bf16_bits_to_f32(w.tensors["mask"])).astype(np.float64))}


# mask boxes: one to five chunks a row; masks read by thread: up to 32 rows
ROWS = [(60, 300, 200, 64), (40, 130, 504, 64), (36, 70, 776, 64), (36, 40, 1288, 64), (150, 20, 304, 64), (60, 31, 1032, 64)]


@pytest.mark.parametrize("fill", FILLS)
@pytest.mark.parametrize("softcap", [0.0, 3.0])
@pytest.mark.parametrize("batch,M,N,K", ROWS)
def test_row_kernel(batch, M, N, K, softcap, fill, cuda_device):
    check(batch, M, N, K, softcap, fill)


# short and long contraction, rows that end inside the kernel's width
CLUSTER = [(20, 130, 1000, 64), (12, 130, 2048, 320), (8, 300, 776, 320), (30, 130, 512, 768)]
FEW = [(1, 40, 200, 64), (4, 64, 1000, 64), (2, 16, 512, 1024), (60, 20, 304, 64)]


@pytest.mark.parametrize("fill", [-1e9, -1e30, LOWEST])
@pytest.mark.parametrize("softcap", [0.0, 3.0])
@pytest.mark.parametrize("batch,M,N,K", CLUSTER + FEW + [(8, 40, 4104, 320)])
def test_other_kernels(batch, M, N, K, softcap, fill, cuda_device):
    check(batch, M, N, K, softcap, fill)


@pytest.mark.parametrize("fill", [-1e9, LOWEST])
def test_unfused(fill, cuda_device):
    check(3, 70, 504, 64, 0.0, fill, fused=False, tol=P.TOL_SOFTMAX_UNFUSED)


def check(batch, M, N, K, softcap, fill, fused=True, tol=P.TOL_SOFTMAX_MAX):
    w = wl.scaled_masked_softmax(batch, M, N, K, seed=M + N, causal=False, softcap=softcap)
    w.tensors["mask"] = finite_mask(M, N, fill)
    got = P.run_gpu(w, P.dev_tensors(w), fused=fused)
    ref = reference(w)
    P.check_outputs(w, got, ref, label=w.name, softmax_tol=tol)
    # rows without a live column, whose probabilities are below that tolerance: one bf16 rounding, and at -1e4 one of the fp32 sum
    # (an ulp is 2^-10 there) in the score and in the reference each
    dead = P.to_f64(got["Y"])[:, 3::4]
    want = ref["Y"][:, 3::4]
    assert (np.abs(dead - want) <= want * (2.0 ** -8 + (2.0 ** -9 if fill == -1e4 else 0.0))).all()


@pytest.mark.parametrize("batch,M,N,causal,sign", [(40, 200, 504, False, 1), (36, 100, 1032, False, 1), (60, 504, 504, True, 1), (40, 200, 504, False, -1),
                                                   (20, 130, 1000, False, 1), (20, 1000, 1000, True, 1), (20, 130, 1000, False, -1), (2, 64, 504, False, 1)])
@pytest.mark.parametrize("fill", [-1e4, -1e9, -1e10, -1e20, -1e30])
def test_scores_far_below_the_others(batch, M, N, causal, sign, fill, cuda_device):
    # the mask folded into the contraction: its last element is 1 in A and, in B, the fill of the columns that are masked
    w = wl.scaled_masked_softmax(batch, M, N, 64, seed=N, causal=causal)
    w.scalars["alpha"] *= sign
    w.tensors["A"][:, :, 63] = wl.f32_to_bf16_bits(np.ones(1, np.float32))
    last = np.zeros(N, np.float32)
    last[64: 200 if N < 1000 else N - 200] = fill * sign  # (whole rows of what a thread holds in the cluster kernel)
    w.tensors["B"][:, 63, :] = wl.f32_to_bf16_bits(last)
    got = P.run_gpu(w, P.dev_tensors(w), fused=True)
    P.check_outputs(w, got, P.run_oracle(w), label=w.name)
