"""The argument-marshalling extension: descriptors read from tensors' shapes and strides, refusals, argument conversions.  Host
only: shapes, strides and addresses of CPU tensors, no call reaches a kernel."""
import os
import subprocess
import sys

import pytest
import torch

import paper_2608_03537_b200 as cf

bf = torch.bfloat16


def _fields(d):
    return {n: getattr(d, n) for n, _ in d._fields_}


@pytest.mark.parametrize("nk", [False, True])
@pytest.mark.parametrize("batch", [None, 1, 3])
def test_descriptor_follows_shapes_and_strides(batch, nk):
    M, N, K = 5, 24, 16
    lead = () if batch is None else (batch,)
    A = torch.zeros(*lead, M, K + 8, dtype=bf)[..., :K]                       # leading dimension K + 8
    B = torch.zeros(*lead, *((N, K + 16) if nk else (K, N)), dtype=bf)[..., : K if nk else N]
    Y, R = torch.zeros(*lead, M, N + 8, dtype=bf)[..., :N], torch.zeros(*lead, M, N, dtype=bf)
    d = cf.make_gemm_desc(A, B, Y, cf.EPI_BIAS_RES_LAYERNORM, residual=R, alpha=2, eps=0.25, fused=[], flags=(cf.FLAG_B_ROW_MAJOR_NK if nk else 0) | cf.FLAG_POST_RELU)
    ldb = K + 16 if nk else N
    want = dict(batch=batch or 1, M=M, N=N, K=K, lda=K + 8, ldb=ldb, ldr=N, ldy=N + 8, batch_stride_a=M * (K + 8), batch_stride_b=(N if nk else K) * ldb,
                batch_stride_r=M * N, batch_stride_y=M * (N + 8), kind=0, mask=0, alpha=2.0, eps=0.25, fused=0,
                flags=(4 if nk else 0) | 1, softcap=0.0, reserved=0)
    assert _fields(d) == want
    d = cf.make_gemm_desc(A, B, Y, cf.EPI_SCALE_MASK_SOFTMAX, mask=cf.MASK_CAUSAL, softcap=1.5, flags=cf.FLAG_B_ROW_MAJOR_NK if nk else 0)
    assert (d.ldr, d.batch_stride_r, d.kind, d.mask, d.softcap, d.fused) == (N, M * N, 2, 1, 1.5, 1)
    assert d.eps == torch.tensor(1e-5).item()


def test_what_the_python_side_refuses():
    A, B, Y = torch.zeros(5, 16, dtype=bf), torch.zeros(16, 24, dtype=bf), torch.zeros(5, 24, dtype=bf)
    for bad in ((A, B.mT, Y), (A, B, Y[:, :16]), (A.mT, B, Y), (torch.zeros(16, 5, dtype=bf).mT, B, Y)):
        with pytest.raises(AssertionError):
            cf.make_gemm_desc(*bad, 0)
    with pytest.raises(IndexError):
        cf.make_gemm_desc(A[0], B, Y, 0)
    for bad, why in (("one", ValueError), ([], TypeError), (None, TypeError)):
        with pytest.raises(why):
            cf.make_gemm_desc(A, B, Y, 0, alpha=bad)
    with pytest.raises(AttributeError):
        cf.gemm_epilogue(A, B, 3, 0)
    W2 = torch.zeros(24, 16, dtype=bf)
    with pytest.raises(AssertionError):
        cf.b2b_mlp_relu(A, B, None, W2, None, torch.zeros(5, 8, dtype=bf))     # O of another width
    with pytest.raises(AssertionError):
        cf.b2b_gemm(A, B, None, torch.zeros(16, 24, dtype=bf).mT, None, Y)      # not dense
    with pytest.raises(ValueError):
        cf.b2b_gemm(A[None], B, None, W2, None, Y)
    with pytest.raises(AssertionError):
        cf.b2b_attention(torch.zeros(2, 5, 16, dtype=bf), torch.zeros(2, 16, 24, dtype=bf), torch.zeros(2, 25, 16, dtype=bf), torch.zeros(2, 5, 16, dtype=bf), alpha=1.0)


def test_scalars_are_taken_as_float_takes_them():
    import numpy as np
    cf.lib()
    A, B, Y = torch.zeros(5, 16, dtype=bf), torch.zeros(16, 24, dtype=bf), torch.zeros(5, 24, dtype=bf)
    for v in (2, 0.25, "0.25", True, np.float32(0.5), np.array(1.5), torch.tensor(3.0)):
        d = cf.make_gemm_desc(A, B, Y, cf.EPI_SCALE_MASK_SOFTMAX, alpha=v, eps=v, softcap=v)
        assert (d.alpha, d.eps, d.softcap) == (float(v),) * 3


ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code, **env):
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT, **env), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]


def test_without_the_extension_only_the_calls_that_need_it_refuse():
    _child("""
import sys
sys.modules["paper_2608_03537_b200._binding"] = None      # as if it had not been built
import torch, paper_2608_03537_b200 as cf
A, B, Y = torch.zeros(5, 16, dtype=torch.bfloat16), torch.zeros(16, 24, dtype=torch.bfloat16), torch.zeros(5, 24, dtype=torch.bfloat16)
d = cf.make_gemm_desc(A, B, Y, cf.EPI_BIAS_RES_LAYERNORM, fused=False)
assert cf.workspace_size(d) == 5 * 24 * 2 and cf.launch_count() == 0
try:
    cf.gemm_epilogue(A, B, Y, cf.EPI_BIAS_RES_LAYERNORM)
except ImportError as e:
    assert "python -m paper_2608_03537_b200.build" in str(e), e
else:
    raise SystemExit("not refused")
""")


def test_a_descriptor_needs_no_library():
    _child("""
import torch, paper_2608_03537_b200 as cf
z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16)
args = [(z(3, 5, 24)[..., :16], z(3, 16, 24), z(3, 5, 24), 0, dict(residual=z(3, 5, 32)[..., :24], flags=1)),
        (z(5, 16), z(24, 16), z(5, 24), 2, dict(mask=1, flags=4, softcap=2, alpha=0.5, fused=[])), (z(5, 16), z(16, 24), z(5, 24), 1, dict(eps=1))]
fields = lambda d: {n: getattr(d, n) for n, _ in d._fields_}
assert cf._bind is None
plain = [fields(cf.make_gemm_desc(*a[:4], **a[4])) for a in args]
assert cf._bind is None
try:
    cf.lib()
except ImportError:
    pass
else:
    raise SystemExit("the library was to be absent")
""".replace("", ""), COMFUSE_LIB="/nonexistent/libcomfuse.so")


def test_both_ways_to_a_descriptor_agree():
    z = lambda *s: torch.zeros(*s, dtype=bf)  # noqa: E731
    native = cf._bound()
    for A, B, Y, kind, kw in ((z(3, 5, 24)[..., :16], z(3, 16, 24), z(3, 5, 24), 0, dict(residual=z(3, 5, 32)[..., :24], flags=1)),
                              (z(5, 16), z(24, 16), z(5, 24), 2, dict(mask=1, flags=4, softcap=2, alpha=0.5, fused=[])),
                              (z(1, 2, 5, 16), z(16, 24), z(5, 24), 1, dict(eps=1))):
        a = _fields(cf.make_gemm_desc(A, B, Y, kind, **kw))
        cf._bind = None
        try:
            b = _fields(cf.make_gemm_desc(A, B, Y, kind, **kw))
        finally:
            cf._bind = native
        assert a == b


def test_the_extension_carries_the_tag_of_its_python():
    import importlib.machinery

    from paper_2608_03537_b200 import build
    tag = importlib.machinery.EXTENSION_SUFFIXES[0]
    assert "cpython" in tag and build.BINDING_PATH.endswith("_binding" + tag)
    assert cf._bound().__file__ == build.BINDING_PATH and not os.path.exists(os.path.join(build.PKG_DIR, "_binding.so"))


class _Recorder:
    """Stands in for comfuse_gemm_spec behind the binding, so that no call reaches the library: what it was given, and INVALID_ARG."""

    def __init__(self):
        import ctypes as c
        proto = c.CFUNCTYPE(c.c_int32, c.c_void_p, c.c_void_p, c.c_void_p, c.c_void_p, c.c_void_p, c.POINTER(c.c_uint64), c.POINTER(c.c_int64),
                            c.POINTER(c.c_uint64), c.c_int32, c.c_void_p, c.c_size_t, c.c_void_p)
        self.seen = []
        self.count = 12
        self.during = lambda: None
        self.fn = proto(self.call)

    def call(self, spec, shape, A, B, Y, params, ld, rows, fused, ws, ws_bytes, stream):
        self.during()
        self.seen.append((params[: self.count], ld[: self.count], rows[:8], stream))
        return cf.ERR_INVALID_ARG

    def __enter__(self):
        import ctypes as c
        L, b = cf.lib(), cf._bound()
        at = lambda f: c.cast(f, c.c_void_p).value  # noqa: E731
        b.bind(at(L.comfuse_gemm_epilogue), at(L.comfuse_b2b_gemm), at(self.fn))
        return self

    def __exit__(self, *exc):
        import ctypes as c
        L = cf.lib()
        cf._bound().bind(*(c.cast(f, c.c_void_p).value for f in (L.comfuse_gemm_epilogue, L.comfuse_b2b_gemm, L.comfuse_gemm_spec)))


class _Stream:
    cuda_stream = 77


def _spec_call(**kw):
    z = lambda *s: torch.zeros(*s, dtype=bf)  # noqa: E731
    spec = cf.make_spec([("acc", -1, -1, -1, 0.0)], 0)
    kw = dict(dict(spec=spec, stream=_Stream()), **kw)
    with pytest.raises(cf.ComfuseError) as e:
        cf.gemm_spec(z(5, 16), z(16, 24), z(5, 24), kw.pop("spec"), **kw)
    assert e.value.status == cf.ERR_INVALID_ARG


def test_parameter_lists_have_a_length_and_are_passed_whole():
    many = [torch.zeros(3, 8, dtype=bf)[:, : 4 + i % 2] if i % 3 else None for i in range(70)]
    with _Recorder() as r:
        r.count = 70
        _spec_call(params=many, row_out=tuple(t for t in many if t is not None))
        params, ld, rows, _ = r.seen.pop()
        assert params == [0 if t is None else t.data_ptr() for t in many] and ld == [0 if t is None else 8 for t in many]
        assert rows == [t.data_ptr() for t in many if t is not None][:8]
        r.count = 12                                 # fewer than a program can name: the others are null
        _spec_call(params={"bias": many[1]}.values())
        assert r.seen.pop()[0] == [many[1].data_ptr()] + [0] * 11
        _spec_call()
        assert r.seen.pop()[:3] == ([0] * 12, [0] * 12, [0] * 8)
        for bad in (dict(params=(t for t in many)), dict(row_out=(t for t in many[1:2])), dict(params=3), dict(row_out=None)):
            with pytest.raises(TypeError):
                _spec_call(**bad)
        assert not r.seen


def test_tensors_of_a_sequence_live_until_the_launch_is_enqueued():
    import gc
    import weakref

    class Fresh:                                     # makes its tensors as it is read
        def __len__(self):
            return 1

        def __getitem__(self, i):
            if i:
                raise IndexError
            t = torch.zeros(24, dtype=bf)
            refs.append(weakref.ref(t))
            return t

    refs, alive = [], []
    with _Recorder() as r:
        r.during = lambda: (gc.collect(), alive.extend(w() is not None for w in refs))
        _spec_call(params=Fresh(), row_out=Fresh())
    assert alive == [True, True]


def test_only_a_program_is_taken_for_a_program():
    import ctypes
    with _Recorder() as r:
        for bad in (cf.make_gemm_shape(1, 5, 24, 16), ctypes.c_int64(0), 0, None):
            with pytest.raises((ctypes.ArgumentError, TypeError)):
                _spec_call(spec=bad)
        assert not r.seen


def test_a_stream_object_may_be_callable():
    class Callable(_Stream):
        def __call__(self):
            return 13

    with _Recorder() as r:
        _spec_call(stream=Callable())
        assert r.seen.pop()[3] == 77


def test_tensors_of_many_dimensions_describe_their_last_two():
    cf._bound()
    one = (1,) * 9
    d = cf.make_gemm_desc(torch.zeros(*one, 5, 16, dtype=bf), torch.zeros(*one, 16, 24, dtype=bf), torch.zeros(*one, 5, 24, dtype=bf), 0)
    assert (d.batch, d.M, d.N, d.K, d.lda, d.ldb, d.ldy) == (1, 5, 24, 16, 16, 24, 24)
