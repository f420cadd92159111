"""Host-only checks of the C-ABI library: it loads, exports every declared symbol, and rejects bad
arguments before launching anything (no GPU needed: every call here fails its argument check)."""
import ctypes as C
import os
import re

import pytest

from paper_2501_00692_b200 import binding as B
from paper_2501_00692_b200.build import build_library

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    build_library()
    return B.lib()


def test_exports_match_header(L):
    hdr = open(os.path.join(ROOT, "include", "adjoint_ssm.h")).read()
    declared = set(re.findall(r"\b(as_[a-z_]+)\s*\(", hdr))
    declared -= {"as_shape_t", "as_params_t", "as_grads_t", "as_dtype_t"}
    assert declared, "no declarations found"
    for name in declared:
        assert hasattr(L, name), f"{name} declared in the header but not exported"
    assert set(B.EXPORTS) == declared
    for name in declared:
        assert name in B.EXPORTS or hasattr(B, name), f"{name} has no Python binding"


def test_version_and_strerror(L):
    assert B.as_version() == 104
    assert B.strerror(0) == "ok"
    assert "tbar" in B.strerror(B.AS_ERR_TBAR)
    assert "unknown" in B.strerror(-999)


def test_struct_layout_matches_c():
    # int32, (pad), int64, 4 x int32  ->  32 bytes with natural alignment
    assert C.sizeof(B.as_shape_t) == 32
    assert B.as_shape_t.seqlen.offset == 8 and B.as_shape_t.d_model.offset == 16 and B.as_shape_t.a_structure.offset == 28
    assert C.sizeof(B.as_params_t) == 48 and C.sizeof(B.as_grads_t) == 48


def test_workspace_query_and_argument_errors(L):
    sh = B.make_shape(2, 65536, 768, 16, B.AS_BF16)
    fwd, grad = B.as_workspace_bytes(sh, 2048)
    assert 0 < fwd < grad < 8 << 30
    for bad, code in ((B.make_shape(0, 8, 64), B.AS_ERR_SHAPE), (B.make_shape(1, 8, 64, 8), B.AS_ERR_SHAPE),
                      (B.make_shape(1, 8, 64, 16, 7), B.AS_ERR_DTYPE), (B.make_shape(1, 8, 60), B.AS_ERR_ALIGN),
                      (B.make_shape(1, 8, 64, 16, B.AS_F32, 5), B.AS_ERR_SHAPE)):
        with pytest.raises(B.AsError) as ei:
            B.as_workspace_bytes(bad, 4)
        assert ei.value.code == code
    with pytest.raises(B.AsError) as ei:
        B.as_workspace_bytes(sh, 0)
    assert ei.value.code == B.AS_ERR_TBAR
    # sizes beyond the 32-bit token-row coordinates or the segment grid dimension are refused, not mis-addressed
    for bad in (B.make_shape(4, 1 << 29, 64), B.make_shape(1, (1 << 31) - 64, 8), B.make_shape(1, 65536 * 2048, 8)):
        with pytest.raises(B.AsError) as ei:
            B.as_workspace_bytes(bad, 4)
        assert ei.value.code == B.AS_ERR_LIMIT
    assert B.as_sm_count() >= 1
    # NULL pointers are rejected before any CUDA call
    p = B.as_params_t(None, None, None, None, None)
    g = B.as_grads_t(None, None, None, None, None, None)
    rc = L.as_adjoint_grad(C.byref(sh), C.byref(p), None, None, 4, 0, C.byref(g), None, 0, None)
    assert rc == B.AS_ERR_NULL
    rc = L.as_ssm_forward(C.byref(sh), C.byref(p), None, None, None, 0, None)
    assert rc == B.AS_ERR_NULL
    # misaligned and undersized workspace (fake, never dereferenced: checks come first)
    ok = C.c_void_p(0x1000)
    p = B.as_params_t(ok, ok, ok, ok, ok)
    g = B.as_grads_t(ok, ok, ok, ok, ok, None)
    assert L.as_adjoint_grad(C.byref(sh), C.byref(p), ok, C.c_void_p(0x1004), 4, 0, C.byref(g), ok, 1 << 40, None) == B.AS_ERR_ALIGN
    assert L.as_adjoint_grad(C.byref(sh), C.byref(p), ok, ok, 4, 0, C.byref(g), ok, 1024, None) == B.AS_ERR_WORKSPACE
    assert L.as_adjoint_grad(C.byref(sh), C.byref(p), ok, ok, 0, 0, C.byref(g), ok, 1 << 40, None) == B.AS_ERR_TBAR
    assert L.as_full_bptt_grad(C.byref(sh), C.byref(p), ok, ok, 0, C.byref(g), ok, 1024, None) == B.AS_ERR_WORKSPACE
    assert L.as_rmsnorm_fwd(C.byref(sh), None, ok, 1e-6, None) == B.AS_ERR_NULL
    # the layers call: same checks, plus the layer count and the limits on layers * batch
    one = B.as_workspace_bytes(sh, 2048)[1]
    many = B.as_workspace_bytes_layers(sh, 4, 2048)
    assert B.as_workspace_bytes_layers(sh, 1, 2048) == one and 3 * one < many < 5 * one
    assert L.as_adjoint_grad_layers(C.byref(sh), 0, C.byref(p), ok, ok, 4, 0, C.byref(g), ok, 1 << 40, None) == B.AS_ERR_SHAPE
    assert L.as_adjoint_grad_layers(C.byref(sh), 3, C.byref(p), ok, ok, 4, 0, C.byref(g), ok, 1024, None) == B.AS_ERR_WORKSPACE
    assert L.as_adjoint_grad_layers(C.byref(sh), 3, C.byref(p), None, ok, 4, 0, C.byref(g), ok, 1 << 40, None) == B.AS_ERR_NULL
    for layers, shape in ((40000, B.make_shape(2, 64, 64)), (1 << 14, B.make_shape(1, 1 << 18, 8))):
        with pytest.raises(B.AsError) as ei:
            B.as_workspace_bytes_layers(shape, layers, 4)
        assert ei.value.code == B.AS_ERR_LIMIT
    # packed weights: size query and argument checks
    assert B.as_wcat_bytes(sh, 3) == 3 * (768 + 32) * 768 * 2 and B.as_wcat_bytes(B.make_shape(0, 8, 64), 1) == 0
    assert L.as_pack_weights(C.byref(sh), 1, C.byref(p), None, None) == B.AS_ERR_NULL
    assert L.as_pack_weights(C.byref(sh), 0, C.byref(p), ok, None) == B.AS_ERR_SHAPE
    f32 = B.make_shape(2, 64, 64)
    assert L.as_pack_weights(C.byref(f32), 1, C.byref(p), ok, None) == B.AS_ERR_DTYPE
    pw = B.as_params_t(ok, ok, ok, ok, ok, C.c_void_p(0x1008))
    assert L.as_adjoint_grad(C.byref(sh), C.byref(pw), ok, ok, 4, 0, C.byref(g), ok, 1 << 40, None) == B.AS_ERR_ALIGN


@pytest.mark.parametrize("shape", [(1, 4100, 248, B.AS_F32), (2, 9000, 512, B.AS_F32), (1, 300, 64, B.AS_F32), (2, 5000, 256, B.AS_BF16)])
def test_forward_refuses_less_scratch_than_reported(L, shape):
    """Neither the kernels nor the result depend on the size of the scratch: one byte short of fwd_bytes is an error, also
    where another form of the contractions could do with less."""
    sh = B.make_shape(*shape[:3], 16, shape[3])
    fwd = B.as_workspace_bytes(sh, shape[1])[0]
    ok = C.c_void_p(0x1000)   # never dereferenced: the size check comes first
    p = B.as_params_t(ok, ok, ok, ok, ok)
    for entry in (L.as_ssm_forward, L.as_ssm_forward_ordered):
        assert entry(C.byref(sh), C.byref(p), ok, ok, ok, 256, None) == B.AS_ERR_WORKSPACE
    assert L.as_ssm_forward(C.byref(sh), C.byref(p), ok, ok, ok, fwd - 1, None) == B.AS_ERR_WORKSPACE


@pytest.mark.parametrize("shape,applies", [((1, 1, 8), 1), ((2, 4096, 64), 1), ((3, 2731, 64), 0), ((1, 65536, 32), 0), ((1, 65536, 72), 1),
                                           ((4, 65536, 128), 1), ((1, 100, 136), 0), ((1, 100, 60), 0), ((0, 100, 64), 0)])
def test_where_a_stack_takes_the_residual_call(L, shape, applies):
    """Narrow fp32 layers, long runs at widths up to 64 apart, which two calls are faster for; bf16 and scalar rates never."""
    assert B.as_ssm_forward_residual_applies(B.make_shape(*shape)) == applies
    assert not B.as_ssm_forward_residual_applies(B.make_shape(*shape, io=B.AS_BF16))
    assert not B.as_ssm_forward_residual_applies(B.make_shape(*shape, a_structure=B.AS_A_SCALAR))


@pytest.mark.parametrize("P,split", [(8, False), (32, False), (56, False), (64, True), (88, True)])
def test_narrow_fp32_gradients_keep_no_split_operands(P, split):
    """From 2^30 multiply-adds on fp32 gradients keep x and the cotangents as three bf16 terms, 12 bytes a value, but not below a width
    of 64, where the tensor-core form is no faster (bytes a token, by a short run that never does, and a long one)."""
    def per_token(T):
        return B.as_workspace_bytes(B.make_shape(1, T, P), 256)[1] / T
    T = (1 << 31) // (P * (P + 32))
    grown = (per_token(T) - per_token(T // 4)) / P
    assert (grown > 4) == split, grown   # the arrays by the segment take less a token in the longer run


def test_missing_library_fails_loudly(monkeypatch):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", "/nonexistent/libadjoint_ssm.so")
    with pytest.raises(RuntimeError, match="no CPU or PyTorch fallback"):
        B.lib()


def test_residual_forward_argument_errors(L):
    sh = B.make_shape(1, 300, 64)
    fwd = B.as_workspace_bytes(sh, 300)[0]
    ok, off = C.c_void_p(0x1000), C.c_void_p(0x1008)   # never dereferenced: the checks come first
    p = B.as_params_t(ok, ok, ok, ok, ok)

    def rc(x=ok, y_in=ok, y_out=ok, yhat=None, ws=ok, ws_bytes=fwd - 1, shape=sh):
        return L.as_ssm_forward_residual(C.byref(shape), C.byref(p), x, y_in, y_out, yhat, 1e-6, ws, ws_bytes, None)

    for one in ("x", "y_in", "y_out", "ws"):
        assert rc(**{one: None}) == B.AS_ERR_NULL, one
    for one in ("x", "y_in", "y_out", "yhat", "ws"):
        assert rc(**{one: off}) == B.AS_ERR_ALIGN, one
    assert rc() == rc(yhat=ok) == B.AS_ERR_WORKSPACE
    for other in (B.make_shape(1, 300, 136), B.make_shape(1, 300, 64, io=B.AS_BF16), B.make_shape(1, 300, 64, a_structure=B.AS_A_SCALAR)):
        assert rc(shape=other, ws_bytes=1 << 40) == B.AS_ERR_LIMIT
