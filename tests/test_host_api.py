"""Host-side checks that need no GPU: the library loads, exports what the header declares,
validates its arguments before touching CUDA, and its host logic agrees with the oracle."""
import ctypes as C
import os
import re

import numpy as np
import pytest

from oracle import rmsmp_oracle as O
from paper_2111_00153_b200 import binding as R
from paper_2111_00153_b200 import build as B
from paper_2111_00153_b200 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _built():
    B.build_library()


def test_library_exports_every_declared_symbol():
    hdr = open(os.path.join(ROOT, "include", "rmsmp.h")).read()
    declared = set(re.findall(r"\b(rmsmp_[a-z0-9_]+)\s*\(", hdr))
    assert declared, "no declarations found"
    assert declared == set(R.EXPORTS)
    lib = R.lib()
    for name in declared:
        assert hasattr(lib, name), name
    for name in R.EXPORTS:
        assert name in declared, name


def test_status_strings():
    seen = {R.rmsmp_status_string(i) for i in range(0, 12)}
    assert len(seen) == 12 and "ok" in seen


def test_assign_rows_matches_oracle_bit_for_bit():
    for idx, (M, K, ratio) in enumerate([(256, 512, (60, 35, 5)), (64, 576, (65, 30, 5)),
                                         (100, 33, (50, 40, 10)), (7, 5, (0, 100, 0)),
                                         (9, 12, (100, 0, 0))]):
        W = synth.weights_normal(synth.rng(90, idx), (M, K))
        s1, b1 = R.rmsmp_assign_rows(W, ratio)
        s2, b2 = O.assign_rows(W, ratio)
        assert np.array_equal(s1, s2) and np.array_equal(b1, b2)
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_assign_rows(np.zeros((4, 4), np.float32), (50, 40, 5))
    assert e.value.status == R.ERR_SHAPE


def test_layer_init_layout():
    scheme = np.array([1, 0, 1, 0, 1, 0, 1], np.uint8)
    bits = np.array([4, 4, 8, 4, 4, 4, 8], np.uint8)
    L = R.rmsmp_layer_init(7, 70, 3, 3, scheme, bits)
    assert (L.nP, L.nF4, L.n8) == (3, 2, 2)
    assert L.Cp == 96 and L.Kp == 896 and L.nblocks == 1     # 9 taps * 96 = 864 -> 896
    offs = [L.off_perm, L.off_slot, L.off_wstep, L.off_alpha, L.off_kind, L.off_blocks, L.off_q4,
            L.off_q8, L.packed_bytes]
    assert all(o % 256 == 0 for o in offs) and offs == sorted(offs)
    assert L.off_q8 - L.off_q4 >= 5 * 896 // 2 and L.packed_bytes - L.off_q8 >= 2 * 896
    L2 = R.rmsmp_layer_init(300, 512, 1, 1, np.ones(300, np.uint8), np.full(300, 4, np.uint8))
    assert L2.nblocks == 3 and L2.Cp == 512 and L2.Kp == 512


def test_layer_init_rejects_bad_input():
    ok_s, ok_b = np.zeros(4, np.uint8), np.full(4, 4, np.uint8)
    for args, err in [((0, 8, 1, 1, ok_s, ok_b), R.ERR_SHAPE),
                      ((4, 0, 1, 1, ok_s, ok_b), R.ERR_SHAPE),
                      ((4, 1000001, 1, 1, ok_s, ok_b), R.ERR_SHAPE),
                      ((4, 8, 17, 1, ok_s, ok_b), R.ERR_SHAPE)]:
        layer = R.rmsmp_layer()
        st = R.lib().rmsmp_layer_init(C.byref(layer), *args[:4], C.c_void_p(args[4].ctypes.data),
                                      C.c_void_p(args[5].ctypes.data))
        assert st == err
    # PoT with 8 bits is not on the method's menu
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_layer_init(4, 8, 1, 1, ok_s, np.array([4, 8, 4, 4], np.uint8))
    assert e.value.status == R.ERR_SCHEME
    with pytest.raises(R.RmsmpError) as e:
        R.rmsmp_layer_init(4, 8, 1, 1, np.array([0, 2, 0, 0], np.uint8), ok_b)
    assert e.value.status == R.ERR_SCHEME
    assert R.lib().rmsmp_layer_init(None, 4, 8, 1, 1, None, None) == R.ERR_NULL


def test_calls_validate_before_any_cuda_work():
    lib = R.lib()
    scheme, bits = np.array([0, 1, 1], np.uint8), np.array([4, 4, 8], np.uint8)
    L = R.rmsmp_layer_init(3, 64, 1, 1, scheme, bits)
    alpha = np.ones(3, np.float32)
    fake = C.c_void_p(0x10000)            # aligned, never dereferenced: validation fails first
    hp = lambda a: C.c_void_p(a.ctypes.data)

    def pack(layer=L, a=alpha, s=scheme, b=bits, dW=fake, dP=fake, nbytes=None, mode=0, layout=0):
        return lib.rmsmp_quantize_pack(dW, layout, C.byref(layer), hp(s), hp(b), hp(a), mode, dP,
                                       layer.packed_bytes if nbytes is None else nbytes, None)

    assert pack(dW=None) == R.ERR_NULL
    assert pack(a=np.array([1, 0, 1], np.float32)) == R.ERR_SCALE
    assert pack(a=np.array([1, np.inf, 1], np.float32)) == R.ERR_SCALE
    assert pack(a=np.array([1, np.nan, 1], np.float32)) == R.ERR_SCALE
    assert pack(a=np.array([1, -2, 1], np.float32)) == R.ERR_SCALE
    assert pack(b=np.array([8, 4, 8], np.uint8)) == R.ERR_SCHEME          # PoT-8
    assert pack(s=np.array([1, 1, 1], np.uint8)) == R.ERR_SCHEME          # differs from layer_init's map
    assert pack(nbytes=16) == R.ERR_BUFFER_TOO_SMALL
    assert pack(dW=C.c_void_p(0x10004)) == R.ERR_ALIGN
    assert pack(dP=C.c_void_p(0x10010)) == R.ERR_ALIGN
    assert pack(layout=1, layer=R.rmsmp_layer()) == R.ERR_BAD_LAYER
    assert pack(mode=7) == R.ERR_SCHEME

    step = C.c_float()
    assert lib.rmsmp_quantize_act(fake, 0, 1.0, 0, fake, C.byref(step), None) == R.ERR_SHAPE
    assert lib.rmsmp_quantize_act(fake, 8, 0.0, 0, fake, C.byref(step), None) == R.ERR_SCALE
    assert lib.rmsmp_quantize_act(None, 8, 1.0, 0, fake, C.byref(step), None) == R.ERR_NULL

    def gemm(N=8, ld=64, act=fake, out=fake, ld_out=3, layout=0, layer=L, packed=fake):
        return lib.rmsmp_gemm(C.byref(layer), packed, act, N, ld, 1.0, out, ld_out, layout, None, None)

    assert gemm(act=None) == R.ERR_NULL
    assert gemm(N=0) == R.ERR_SHAPE
    assert gemm(ld=48) == R.ERR_SHAPE          # shorter than K
    assert gemm(ld=72) == R.ERR_ALIGN          # not a multiple of 16
    assert gemm(ld_out=2) == R.ERR_SHAPE
    assert gemm(layout=1, ld_out=7) == R.ERR_SHAPE
    assert gemm(act=C.c_void_p(0x10001)) == R.ERR_ALIGN
    assert gemm(layer=R.rmsmp_layer()) == R.ERR_BAD_LAYER
    Lc = R.rmsmp_layer_init(3, 16, 3, 3, scheme, bits)
    assert gemm(layer=Lc) == R.ERR_SHAPE       # a conv layer is not a linear layer

    def conv(B=1, H=8, W=8, stride=1, pad=1, act=fake, layer=Lc):
        return lib.rmsmp_conv_implicit(C.byref(layer), fake, act, B, H, W, stride, pad, 1.0, fake, 0,
                                       None, None)

    assert conv(B=0) == R.ERR_SHAPE
    assert conv(stride=0) == R.ERR_SHAPE
    assert conv(H=1, pad=0) == R.ERR_SHAPE     # kernel larger than padded image
    assert conv(act=None) == R.ERR_NULL
    assert lib.rmsmp_last_device_status(None, None) == R.ERR_NULL


def test_no_gpu_means_loud_failure_not_fallback():
    import torch
    if torch.cuda.is_available():
        pytest.skip("GPU present")
    lib = R.lib()
    step = C.c_float()
    st = lib.rmsmp_quantize_act(C.c_void_p(0x10000), 16, 1.0, 0, C.c_void_p(0x20000), C.byref(step), None)
    assert st in (R.ERR_CUDA, R.ERR_ARCH)


def test_marshalled_calls_take_the_python_signatures_and_raise_like_them():
    """The calls of the extension module without a GPU: positional and keyword arguments, defaults, argument errors as
    TypeError, the library's own refusals as RmsmpError with their status."""
    good = R.rmsmp_layer_init(4, 16, 1, 1, np.zeros(4, np.uint8), np.full(4, 4, np.uint8))
    args = (good, 256, 256, 1, 16, 0.5, 256, 4)
    for bad_call, status in (
            (lambda: R.rmsmp_gemm(good, None, 256, 1, 16, 0.5, 256, 4, stream=0), R.ERR_NULL),
            (lambda: R.rmsmp_gemm(R.rmsmp_layer(), *args[1:], stream=0), R.ERR_BAD_LAYER),
            (lambda: R.rmsmp_gemm(layer=good, d_packed=256, d_act=256, N=1, ld_act=8, act_step=0.5, d_out=256, ld_out=4, stream=0), R.ERR_SHAPE),
            (lambda: R.rmsmp_gemm(*args, 7, None, 0), R.ERR_SHAPE),
            (lambda: R.rmsmp_gemm(good, 256, 257, *args[3:], stream=0), R.ERR_ALIGN),
            (lambda: R.rmsmp_gemm(*args[:5], float("inf"), 256, 4, stream=0), R.ERR_SCALE),
            (lambda: R.rmsmp_gemm_workspace(good, 256, None, *args[2:], stream=0), R.ERR_NULL),
            (lambda: R.rmsmp_expand_weights(good, 256, 256, 1, stream=0), R.ERR_BUFFER_TOO_SMALL),
            (lambda: R.rmsmp_quantize_act(256, 0, 3.0, R.ACT_U4, 256, stream=0), R.ERR_SHAPE),
            (lambda: R.rmsmp_quantize_act(256, 4, -3.0, R.ACT_U4, 256, stream=0), R.ERR_SCALE),
            (lambda: R.rmsmp_conv_implicit(good, 256, 256, 1, 4, 4, 0, 0, 0.5, 256, stream=0), R.ERR_SHAPE),
            (lambda: R.rmsmp_im2col_codes(256, 1, 4, 4, 3, 2, 3, 3, 1, 1, 256, 32, stream=0), R.ERR_SHAPE),
            (lambda: R.rmsmp_gemm_grouped_launch(R.rmsmp_grouped_plan(), stream=0), R.ERR_BAD_LAYER)):
        with pytest.raises(R.RmsmpError) as e:
            bad_call()
        assert e.value.status == status
    for bad_call in (lambda: R.rmsmp_gemm(good), lambda: R.rmsmp_gemm(*args, nonsense=1), lambda: R.rmsmp_gemm(*args, d_out=1),
                     lambda: R.rmsmp_gemm(1, *args[1:], stream=0), lambda: R.rmsmp_gemm(R.rmsmp_grouped_plan(), *args[1:], stream=0),
                     lambda: R.rmsmp_gemm(*args[:3], 1.5, *args[4:], stream=0), lambda: R.rmsmp_gemm(*args, 0, None, 0, 0)):
        with pytest.raises(TypeError):
            bad_call()
    with pytest.raises(OverflowError):
        R.rmsmp_conv_implicit(good, 256, 256, 1 << 40, 4, 4, 1, 0, 0.5, 256, stream=0)


@pytest.mark.parametrize("convert", [lambda a: a, list, lambda a: a.astype(np.int64), lambda a: np.repeat(a, 2)[::2]],
                         ids=["array", "list", "int64", "strided"])
def test_marshalled_pack_takes_any_host_array(convert):
    """Scheme, precision and scale per row as what numpy makes an array of; refusals come from the library."""
    scheme, bits, alpha = np.array([0, 1, 1, 1], np.uint8), np.array([4, 4, 8, 4], np.uint8), np.full(4, 3, np.float32)
    layer = R.rmsmp_layer_init(4, 16, 1, 1, scheme, bits)

    def call(s=scheme, b=bits, a=alpha, mode=R.POT_NEAREST, packed=256, nbytes=1 << 20):
        R.rmsmp_quantize_pack(256, R.W_LINEAR, layer, convert(s), convert(b), convert(a), mode, packed, nbytes, stream=0)
    for kw, status in ((dict(s=np.zeros(4, np.uint8)), R.ERR_SCHEME), (dict(b=np.array([4, 4, 5, 4], np.uint8)), R.ERR_SCHEME),
                       (dict(a=alpha * 0), R.ERR_SCALE), (dict(mode=9), R.ERR_SCHEME), (dict(packed=None), R.ERR_NULL),
                       (dict(packed=264), R.ERR_ALIGN), (dict(nbytes=16), R.ERR_BUFFER_TOO_SMALL)):
        with pytest.raises(R.RmsmpError) as e:
            call(**kw)
        assert e.value.status == status
    with pytest.raises(ValueError):
        call(a=alpha[:3])
    with pytest.raises((TypeError, ValueError)):
        R.rmsmp_quantize_pack(256, R.W_LINEAR, layer, "abc", bits, alpha, R.POT_NEAREST, 256, 1 << 20, stream=0)


def test_marshalling_module_is_named_for_its_interpreter():
    import sysconfig
    assert os.path.basename(B.MARSHAL) == "_marshal" + sysconfig.get_config_var("EXT_SUFFIX")
    assert os.path.exists(B.MARSHAL) and not os.path.exists(os.path.join(os.path.dirname(B.MARSHAL), "_marshal.so"))


def test_names_are_there_without_the_library_and_calls_say_what_is_missing():
    import subprocess
    import sys
    code = """
from paper_2111_00153_b200 import binding as R
R.LIB_PATH = "/nonexistent/librmsmp.so"
from paper_2111_00153_b200.binding import rmsmp_gemm, rmsmp_workspace_bytes
assert hasattr(R, "rmsmp_quantize_act") and not hasattr(R, "rmsmp_no_such_call")
for call in (rmsmp_gemm, R.rmsmp_quantize_act):
    try:
        call()
    except RuntimeError as e:
        assert "is missing" in str(e)
    else:
        raise SystemExit("no error")
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stdout + r.stderr


def test_read_only_loads_go_through_pointers_ordered_behind_the_wait():
    """To the compiler a read-only load is a function of its address: in a kernel that waits for the one in front, its
    pointer must not exist before the wait.  Kernels take their problem by value, so a load straight through a member of
    it is what must not be there (a local copy whose pointers were ordered may)."""
    direct = re.compile(r"__ldg\((?:reinterpret_cast<[^>]*>\()?\s*([pa])\.(\w+)")
    for name in sorted(os.listdir(B.CSRC)):
        if not name.endswith(".cu") or name in ("stream.cu",):          # (its table's and packed codes' early reads are the rule's exemption)
            continue
        text = open(os.path.join(B.CSRC, name)).read()
        if "pdl_wait()" not in text:
            continue
        for obj, member in direct.findall(text):
            ordered = re.search(r"%s\.%s = pdl_ordered\(%s\.%s\)" % (obj, member, obj, member), text)
            from_table = name == "simt.cu" and (obj, member) == ("p", "perm")      # (a problem read from the launch's table)
            assert ordered or from_table, (name, obj, member)
