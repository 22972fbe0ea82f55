"""What users have this library do, as cases that can be timed and compared.

Every case goes through the public Python entry points of ``paper_2608_03537_b200`` with device tensors (one with host
tensors).  A user's program keeps the weights, the workspace and the output buffer and calls the same function for every step, so
``prepare`` makes those and ``run`` is one call.  Values: activations and attention operands N(0, 1), weights
N(0, 1 / fan-in), biases U(-0.1, 0.1), gains N(1, 0.02), all bf16.
"""
import math

import torch

import paper_2608_03537_b200 as cf


def listed():
    return [
        # post-norm block of a very small model: launch and call latency is all there is
        {"name": "post_norm_tiny", "path": "norm", "M": 256, "N": 256, "K": 256, "nk": False, "residual": True, "affine": False, "relu": False},
        # BERT-base FFN output + residual + LayerNorm, 16 sequences of 512 tokens
        {"name": "post_norm_bert_ffn", "path": "norm", "M": 8192, "N": 768, "K": 3072, "nk": False, "residual": True, "affine": True, "relu": False},
        # wide linear layer with GELU, residual, RMSNorm and the row's maximum: prefill
        {"name": "complex_prefill", "path": "complex", "M": 8192, "N": 4096, "K": 4096, "nk": False, "residual": True, "activation": True},
        # the same layer for the tokens of one decoding step, weight stored [out, in] as a linear layer keeps it
        {"name": "complex_decode", "path": "complex", "M": 40, "N": 4096, "K": 4096, "nk": True, "residual": True, "activation": True},
        # causal attention probabilities, 64 batch x heads of 2048 positions
        {"name": "softmax_causal", "path": "softmax", "batch": 64, "M": 2048, "N": 2048, "K": 64, "mask": "causal", "softcap": 0.0, "nk": False},
        # attention probabilities with a padded, position-biased additive mask, 8 sequences x 12 heads, keys one per row
        {"name": "softmax_masked", "path": "softmax", "batch": 96, "M": 504, "N": 504, "K": 64, "mask": "additive", "softcap": 0.0, "nk": True},
        # narrow transformer MLP with its residual and LayerNorm
        {"name": "mlp_gelu_norm", "path": "mlp", "M": 32768, "N1": 512, "affine": False},
        # 4096 target positions attend to 256 source positions
        {"name": "target_attention", "path": "attention", "batch": 32, "M": 4096, "S": 256, "nk": False},
        # self-attention over 512 positions, keys one per row
        {"name": "self_attention", "path": "attention", "batch": 256, "M": 512, "S": 512, "nk": True},
        # bottom MLP of a recommendation model, 1024 -> 512 -> 128
        {"name": "dlrm_bottom_mlp", "path": "relu_mlp", "M": 32768, "K": 1024, "N1": 512},
        # an epilogue given as a node list that no built-in op list covers
        {"name": "program_range_normalise", "path": "program", "program": "range_normalise", "M": 8192, "N": 1024, "K": 1024, "nk": False},
        # the BERT-base case with activations, residual and result in pinned host memory
        {"name": "post_norm_bert_ffn_host", "path": "norm_host", "M": 8192, "N": 768, "K": 3072, "affine": True},
    ]


def _log(rng, lo, hi, step=1):
    """An integer multiple of `step` in [lo, hi], spread evenly over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / step)) * step))


def draw(rng):
    path = rng.choice(["norm", "norm", "complex", "complex", "softmax", "softmax", "mlp", "attention", "attention", "relu_mlp", "program", "norm_host"])
    flag = lambda: rng.random() < 0.5  # noqa: E731
    if path == "norm":
        return {"path": path, "M": _log(rng, 1, 8192), "N": _log(rng, 256, 4096, 8), "K": _log(rng, 64, 4096, 8), "nk": flag(), "residual": flag(),
                "affine": flag(), "relu": flag()}
    if path == "complex":
        return {"path": path, "M": _log(rng, 1, 8192), "N": _log(rng, 256, 4096, 8), "K": _log(rng, 64, 4096, 8), "nk": flag(), "residual": flag(),
                "activation": flag()}
    if path == "softmax":
        mask = rng.choice(["none", "causal", "additive"])
        n = _log(rng, 64, 2048, 8)
        m = n if mask == "causal" else _log(rng, 16, 2048)
        batch = _log(rng, 1, max(1, min(64, (1 << 27) // (m * n))))
        return {"path": path, "batch": batch, "M": m, "N": n, "K": rng.choice([32, 64, 64, 72, 128]), "mask": mask, "softcap": rng.choice([0.0, 0.0, 30.0]),
                "nk": flag()}
    if path == "mlp":
        return {"path": path, "M": _log(rng, 1, 32768), "N1": _log(rng, 128, 1024, 8), "affine": flag()}
    if path == "attention":
        m = _log(rng, 16, 4096)
        return {"path": path, "batch": _log(rng, 1, max(1, min(256, 131072 // m))), "M": m, "S": _log(rng, 8, 512, 8), "nk": flag()}
    if path == "relu_mlp":
        return {"path": path, "M": _log(rng, 1, 32768), "K": _log(rng, 64, 1024, 8), "N1": _log(rng, 64, 512, 8)}
    if path == "program":
        return {"path": path, "program": rng.choice(["range_normalise", "gated_minmax"]), "M": _log(rng, 1, 8192), "N": rng.choice([256, 512, 768, 1024, 1536, 2048]),
                "K": _log(rng, 64, 2048, 8), "nk": flag()}
    return {"path": path, "M": _log(rng, 256, 8192), "N": _log(rng, 256, 1024, 8), "K": _log(rng, 64, 3072, 8), "affine": flag()}


# Epilogues as node lists: (op, input, input, parameter slot, immediate).  Slot 0 is the bias.
class _Nodes(list):
    def add(self, op, a=-1, b=-1, param=-1, imm=0.0):
        self.append((op, a, b, param, imm))
        return len(self) - 1


def _range_normalise():
    """x = acc + bias rescaled to its row's range; the row's minimum and maximum, a product over the row, the result's sum and arg max as row outputs."""
    g = _Nodes()
    x = g.add("add", g.add("acc"), g.add("rowvec", param=0))
    lo, hi = g.add("rmin", x), g.add("rmax", x)
    y = g.add("div", g.add("sub", x, lo), g.add("add", g.add("sub", hi, lo), g.add("const", imm=1e-3)))
    pr = g.add("prod", g.add("add", g.add("mul", g.add("sigmoid", x), g.add("const", imm=0.01)), g.add("const", imm=0.995)))
    return g, y, (lo, hi, pr, g.add("sum", y), g.add("argmax", y))


def _gated_minmax():
    """x * sigmoid(x), x = acc + bias, rescaled to its row's range; the row's minimum and maximum as row outputs."""
    g = _Nodes()
    x = g.add("add", g.add("acc"), g.add("rowvec", param=0))
    s = g.add("mul", x, g.add("sigmoid", x))
    lo, hi = g.add("rmin", s), g.add("rmax", s)
    y = g.add("div", g.add("sub", s, lo), g.add("add", g.add("sub", hi, lo), g.add("const", imm=1e-3)))
    return g, y, (lo, hi)


_PROGRAMS = {"range_normalise": _range_normalise, "gated_minmax": _gated_minmax}
_KINDS = {"norm": cf.EPI_BIAS_RES_LAYERNORM, "norm_host": cf.EPI_BIAS_RES_LAYERNORM, "complex": cf.EPI_BIAS_GELU_RES_RMSNORM_MAX,
          "softmax": cf.EPI_SCALE_MASK_SOFTMAX}


class _Make:
    """bf16 device tensors from one seeded generator."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(self, *shape, mean=0.0, std=1.0):
        return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(mean, std, generator=self.g).to(torch.bfloat16)

    def uniform(self, n, lo=-0.1, hi=0.1):
        return torch.empty(n, dtype=torch.float32, device="cuda").uniform_(lo, hi, generator=self.g).to(torch.bfloat16)

    def weight(self, k, n, nk=False):
        return self.normal(*((n, k) if nk else (k, n)), std=k ** -0.5)


def _workspace(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda") if nbytes else None


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    c, mk, path = case, _Make(seed), case["path"]
    out = lambda *shape: torch.empty(shape, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    s = {"case": c, "path": path}
    if path in ("norm", "complex", "norm_host"):
        M, N, K = c["M"], c["N"], c["K"]
        nk = c.get("nk", False)
        s["A"], s["B"], s["Y"] = mk.normal(M, K), mk.weight(K, N, nk), out(M, N)
        kw = {"bias": mk.uniform(N), "residual": mk.normal(M, N) if c.get("residual", True) else None, "flags": cf.FLAG_B_ROW_MAJOR_NK if nk else 0}
        if path == "complex":
            kw["gamma"] = mk.normal(N, mean=1.0, std=0.02)
            kw["row_max"] = torch.empty(M, dtype=torch.float32, device="cuda")
            kw["row_argmax"] = torch.empty(M, dtype=torch.int32, device="cuda")
            kw["flags"] |= 0 if c["activation"] else cf.FLAG_NO_ACTIVATION
        else:
            if c["affine"]:
                kw["gamma"], kw["beta"] = mk.normal(N, mean=1.0, std=0.02), mk.normal(N, std=0.02)
            kw["flags"] |= cf.FLAG_POST_RELU if c.get("relu", False) else 0
        desc = cf.make_gemm_desc(s["A"], s["B"], s["Y"], _KINDS[path], residual=kw["residual"], flags=kw["flags"])
        kw["workspace"] = _workspace(cf.workspace_size(desc))
        if path == "norm_host":
            mask = cf.HOST_A | cf.HOST_RESIDUAL | cf.HOST_Y
            kw.update(host_mask=mask, staging=_workspace(cf.host_staging_size(desc, mask)), residual=_pinned(kw["residual"]))
            s["A"], s["Y"] = _pinned(s["A"]), torch.empty(M, N, dtype=torch.bfloat16, pin_memory=True)
        s["kw"] = kw
    elif path == "softmax":
        b, M, N, K = c["batch"], c["M"], c["N"], c["K"]
        s["A"], s["B"], s["Y"] = mk.normal(b, M, K), mk.normal(b, *((N, K) if c["nk"] else (K, N))), out(b, M, N)
        kw = {"alpha": K ** -0.5, "softcap": c["softcap"], "flags": cf.FLAG_B_ROW_MAJOR_NK if c["nk"] else 0}
        if c["mask"] == "causal":
            kw["mask"] = cf.MASK_CAUSAL
        elif c["mask"] == "additive":  # distance bias plus a learned term; the last positions are padding
            i, j = torch.arange(M, device="cuda")[:, None], torch.arange(N, device="cuda")[None, :]
            bias = (i - j).abs().float() * (-1.0 / 32) + mk.normal(M, N).float() * 0.5
            kw["mask"], kw["mask_tensor"] = cf.MASK_ADDITIVE, bias.masked_fill(j >= N - N // 10, -math.inf).to(torch.bfloat16).contiguous()
        s["kw"] = kw
    elif path == "mlp":
        M, d, N1 = c["M"], 128, c["N1"]
        s["args"] = [mk.normal(M, d), mk.weight(d, N1), mk.uniform(N1), mk.weight(N1, d), mk.uniform(d), out(M, d)]
        s["kw"] = {"gamma": mk.normal(d, mean=1.0, std=0.02), "beta": mk.normal(d, std=0.02)} if c["affine"] else {}
    elif path == "relu_mlp":
        M, K, N1 = c["M"], c["K"], c["N1"]
        s["args"] = [mk.normal(M, K), mk.weight(K, N1), mk.uniform(N1), mk.weight(N1, 128), mk.uniform(128), out(M, 128)]
    elif path == "attention":
        b, M, S, d = c["batch"], c["M"], c["S"], 128
        s["args"] = [mk.normal(b, M, d), mk.normal(b, *((S, d) if c["nk"] else (d, S))), mk.normal(b, S, d), out(b, M, d)]
        s["kw"] = {"alpha": d ** -0.5, "keys_row_major": c["nk"]}
    elif path == "program":
        M, N, K, nk = c["M"], c["N"], c["K"], c["nk"]
        nodes, terminal, row_outputs = _PROGRAMS[c["program"]]()
        s["spec"] = cf.make_spec(nodes, terminal, 1, row_outputs)
        s["A"], s["B"], s["Y"] = mk.normal(M, K), mk.weight(K, N, nk), out(M, N)
        shape = cf.make_gemm_shape(1, M, N, K, flags=cf.FLAG_B_ROW_MAJOR_NK if nk else 0)
        cf.gemm_spec_prepare(s["spec"], shape, 1)
        s["kw"] = {"params": [mk.uniform(N)], "b_nk": nk, "workspace": _workspace(cf.gemm_spec_workspace_size(s["spec"], shape, True)),
                   "row_out": [torch.empty(M, dtype=torch.int32 if nodes[r][0] == "argmax" else torch.float32, device="cuda") for r in row_outputs]}
    return s


def run(state):
    s, path = state, state["path"]
    if path in ("norm", "softmax"):
        return cf.gemm_epilogue(s["A"], s["B"], s["Y"], _KINDS[path], **s["kw"])
    if path == "complex":
        return cf.gemm_epilogue(s["A"], s["B"], s["Y"], _KINDS[path], **s["kw"]), s["kw"]["row_max"], s["kw"]["row_argmax"]
    if path == "norm_host":
        return cf.gemm_epilogue_host(s["A"], s["B"], s["Y"], _KINDS[path], **s["kw"])
    if path == "mlp":
        return cf.b2b_gemm(*s["args"], **s["kw"])
    if path == "relu_mlp":
        return cf.b2b_mlp_relu(*s["args"])
    if path == "attention":
        return cf.b2b_attention(*s["args"], **s["kw"])
    return cf.gemm_spec(s["A"], s["B"], s["Y"], s["spec"], **s["kw"]), s["kw"]["row_out"]


def work(case):
    c, path = case, case["path"]
    if path in ("norm", "complex", "norm_host", "program"):
        M, N, K = c["M"], c["N"], c["K"]
        has_residual = path != "program" and c.get("residual", True)
        vectors = 2 if path == "complex" else 3 if c.get("affine") else 1
        row_outputs = {"complex": 2, "program": 5 if c.get("program") == "range_normalise" else 2}.get(path, 0)
        return {"bytes": 2 * (M * K + K * N + M * N * (2 if has_residual else 1) + vectors * N) + 4 * M * row_outputs, "flops": 2 * M * N * K}
    if path == "softmax":
        b, M, N, K = c["batch"], c["M"], c["N"], c["K"]
        live = (M + 1) / (2 * M) if c["mask"] == "causal" else 1.0
        return {"bytes": 2 * (b * (M * K + K * N + M * N) + (M * N if c["mask"] == "additive" else 0)), "flops": 2 * b * M * N * K * live}
    if path == "attention":
        b, M, S = c["batch"], c["M"], c["S"]
        return {"bytes": 2 * b * 128 * (2 * M + 2 * S), "flops": 4 * b * M * S * 128}
    M, K, N1 = c["M"], c.get("K", 128), c["N1"]
    vectors = N1 + 128 + (256 if c.get("affine") else 0)
    return {"bytes": 2 * (M * K + K * N1 + N1 * 128 + M * 128 + vectors), "flops": 2 * M * N1 * (K + 128)}


def tolerance(case):
    # Against the same calls in 64 bits every path shows a relative error of 1.5e-3 (one bf16 rounding) to 2.3e-3 (a bf16 intermediate too),
    # and up to 1 row in 1000 whose two largest values are so close that the arg max differs.
    return {"rel": 1e-2, "differ": 5e-3}
