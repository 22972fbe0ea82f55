"""Fused kinds behind a GEMM of few rows (weights as the tensor core's 128-row operand, contraction split over a
cluster), at the edges of its cuts: one row, full and partial row groups of 16 / 32 / 64, full and partial 128-column tiles,
one and two tiles per CTA, 1 to 8 shares of the contraction, row slices that end empty, the two-kernel form with a partial last
block, both sides of the lines that follow what the L2 delivers, both storage orders of the weights.  Against the fp64 oracle with the bounds of the other fused forms."""
import pytest
import torch

import paper_2608_03537_b200 as cf
import workloads as wl
from tests import parity as P

pytestmark = pytest.mark.gpu

SHAPES = [(1, 8, 8), (16, 128, 64), (17, 136, 768), (32, 256, 72), (33, 2056, 200), (63, 1000, 2056), (64, 1024, 1792), (65, 4096, 64),
          (2, 264, 4104), (40, 4096, 4096), (5, 2048, 1024), (70, 2824, 1032), (300, 768, 768), (900, 520, 320), (2112, 520, 1032), (2369, 520, 1032), (1100, 512, 1544),
          (7110, 24, 2568), (4740, 8, 776)]


@pytest.mark.parametrize("nk", [False, True])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_few_rows(M, N, K, nk, cuda_device):
    flags = cf.FLAG_B_ROW_MAJOR_NK if nk else 0
    for w in (wl.post_norm(M, N, K, seed=M + N + K, affine=True, relu=bool(M & 1)), wl.complex_subgraph(M, N, K, seed=M + N, activation=not (M & 1))):
        T = P.dev_tensors(w)
        ln = w.kind == wl.KIND_BIAS_RES_LAYERNORM
        B = T["B"].mT.contiguous() if nk else T["B"]
        Y = P.guarded((M, N), torch.bfloat16, float("nan"), T["A"].device)
        got = {"Y": Y}
        kw = dict(bias=T["bias"], residual=T["residual"], gamma=T["gamma"], alpha=w.scalars["alpha"], eps=w.scalars["eps"])
        if ln:
            kw.update(beta=T["beta"], flags=flags | (cf.FLAG_POST_RELU if w.scalars.get("relu") else 0))
        else:
            got["row_max"] = kw["row_max"] = P.guarded((M,), torch.float32, float("nan"), T["A"].device)
            got["row_argmax"] = kw["row_argmax"] = P.guarded((M,), torch.int32, -1, T["A"].device)
            kw["flags"] = flags | (0 if w.scalars.get("activation", True) else cf.FLAG_NO_ACTIVATION)
        kind = cf.EPI_BIAS_RES_LAYERNORM if ln else cf.EPI_BIAS_GELU_RES_RMSNORM_MAX
        desc = cf.make_gemm_desc(T["A"], B, Y, kind, residual=T["residual"], flags=kw["flags"])
        ws = P.guarded((max(16, cf.workspace_size(desc)),), torch.uint8, 0xEE, T["A"].device)
        for _ in range(2):
            cf.gemm_epilogue(T["A"], B, Y, kind, workspace=ws, **kw)
        torch.cuda.synchronize()
        P.check_canaries({"ws": ws, **got}, label=w.name)
        ref = P.run_oracle(w)
        ymax = float(abs(ref["Y"]).max())
        bounds = {"norm_tol": P.TOL_NORM_MAX if ymax < 8.0 else 2.0 ** -7 * ymax}   # bf16 half-ulp of the largest magnitude, twice
        if not ln:
            if cf.workspace_size(desc) > 0:
                bounds["rowmax_tol"] = 3e-2   # the two-kernel form takes the maximum from values that went through fp16
        P.check_outputs(w, got, ref, label=f"{w.name} nk={nk}", **bounds)


@pytest.mark.parametrize("mask", ["none", "causal", "additive"])
@pytest.mark.parametrize("batch,M,N,K,softcap", [(1, 1, 8, 8, 0.0), (3, 16, 128, 64, 0.0), (2, 17, 136, 72, 3.0), (5, 33, 1000, 64, 0.0), (1, 65, 2056, 64, 0.0), (2, 64, 2048, 776, 2.5),
                                                 (1, 40, 4096, 2056, 0.0), (30, 130, 120, 64, 0.0)])
def test_few_rows_softmax(batch, M, N, K, softcap, mask, cuda_device):
    import numpy as np
    if mask == "causal":
        N = M = min(M * 8, 520)
    w = wl.scaled_masked_softmax(batch, M, N, K, seed=M + N, causal=mask == "causal", softcap=softcap)
    if mask == "additive":
        g = np.random.default_rng(N)
        m = (g.standard_normal((M, N)) * 2.0).astype(np.float32)
        m[g.random((M, N)) < 0.2] = -np.inf
        m[M // 2, :] = -np.inf                     # a row without a live column is all zero
        m[0, : N // 2] = -np.inf                   # a row whose first column ranges have none
        w.tensors["mask"] = wl.f32_to_bf16_bits(m)
    got = P.run_gpu(w, P.dev_tensors(w), fused=True)
    P.check_outputs(w, got, P.run_oracle(w), label=f"{w.name} {mask}", softmax_tol=P.TOL_SOFTMAX_MAX)
    if mask == "additive":
        assert (got["Y"][:, M // 2, :] == 0).all()


@pytest.mark.parametrize("batch,M,N,K", [(3, 64, 1000, 320), (2, 5, 72, 776), (1, 40, 2056, 64), (4, 17, 512, 64)])
def test_softmax_rows_with_a_nan_are_nan(batch, M, N, K, cuda_device):
    bf = torch.bfloat16
    g = torch.Generator(device=cuda_device).manual_seed(N)
    A, B = (torch.empty(s, device=cuda_device).normal_(generator=g).to(bf) for s in ((batch, M, K), (batch, K, N)))
    A[:, 1, 3] = float("nan")                            # every score of row 1
    mask = torch.zeros(M, N, dtype=bf, device=cuda_device)
    mask[2, N - 1] = float("nan")                        # one score of row 2
    mask[3, : N - 8] = float("-inf")
    mask[3, N - 3] = float("nan")                        # ... of row 3, whose other column ranges have no live column
    mask[4, 0] = float("inf")
    for m in (None, mask):
        Y = torch.zeros(batch, M, N, dtype=bf, device=cuda_device)
        cf.gemm_epilogue(A, B, Y, cf.EPI_SCALE_MASK_SOFTMAX, alpha=K ** -0.5, mask=cf.MASK_NONE if m is None else cf.MASK_ADDITIVE, mask_tensor=m)
        want = torch.zeros(M, dtype=torch.bool, device=cuda_device)
        want[1 : 2 if m is None else 5] = True
        assert torch.equal(Y.isnan(), want[None, :, None].expand_as(Y))
