"""The FP32 tensor-core kernels without a GPU: they compile for sm_103a, and what the
accuracy tests ask of them is sharp enough."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import f32split
import oracle

from paper_0911_3456_gb300 import _capi as C


@pytest.mark.parametrize("shape,spec,ok", [
    (((64, 64, 4), (16, 3, 3, 4)), "f32tc", True),
    (((40, 50, 33), (7, 13, 13, 33)), "f32tc", True),
    (((128, 128, 8), (16, 9, 9, 8)), "f32tc:nt=64,r=4,gc=8,jt=9,ru=2", True),
    (((128, 128, 8), (16, 9, 9, 8)), "f32tc:nt=64,r=4,gc=8,jt=9", False),
])
def test_rtcg_check(shape, spec, ok):
    log = ctypes.create_string_buffer(8192)
    st = C.load().fbcorr_rtcg_check(C.I64_3(*shape[0]), C.I64_4(*shape[1]), C.epilogue((0.0, 1.0)), spec.encode(), log,
                                    len(log))
    assert (st == 0) == ok, log.value.decode()


@pytest.mark.parametrize("fields", ["nt=64,r=4,gc=8,jt=0,ru=2", "nt=64,r=4,gc=8,jt=9,ru=0", "nt=64,r=4,gc=0,jt=9,ru=2",
                                    "nt=0,r=4,gc=8,jt=9,ru=2", "nt=64,r=0,gc=8,jt=9,ru=2", "nt=-64,r=4,gc=8,jt=9,ru=2",
                                    "nt=64,r=4,gc=8,jt=-1,ru=2", "nt=64,r=-4,gc=8,jt=9,ru=2", "nt=64,r=4,gc=-8,jt=9,ru=2",
                                    "nt=64,r=4,gc=8,jt=9,ru=-2", "nt=96,r=4,gc=8,jt=9,ru=2", "nt=72,r=4,gc=8,jt=9,ru=2",
                                    "nt=64,r=5,gc=8,jt=9,ru=2", "nt=64,r=268435456,gc=8,jt=9,ru=2", "nt=64,r=4,gc=12,jt=9,ru=2",
                                    "nt=64,r=4,gc=8,jt=10,ru=2", "nt=64,r=4,gc=8,jt=2000000000,ru=2",
                                    "nt=64,r=4,gc=8,jt=9,ru=13", "nt=64,r=4,gc=8,jt=9,ru=2000000000"])
def test_rtcg_check_refuses_tiles_that_no_plan_takes(fields):
    """In a child process: a tile of zeros once divided by zero on the host."""
    code = ("from paper_0911_3456_gb300 import _capi as C; "
            "print(C.load().fbcorr_rtcg_check(C.I64_3(128, 128, 8), C.I64_4(16, 9, 9, 8), C.epilogue(None), "
            f"b'f32tc:{fields}', None, 0))")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and r.stdout.strip() == "3", r.stderr       # FBCORR_ERR_UNSUPPORTED


def _kernels(directory):
    text = "".join(f.read_text() for f in directory.iterdir())
    return {name for name in ("fbc_f32tc_", "fbc_f32dw_", "fbc_batch(") if f") {name}" in text}, text


def test_rtcg_check_compiles_the_kernels_of_all_three_passes(tmp_path, monkeypatch):
    monkeypatch.setenv("FBCORR_DUMP_DIR", str(tmp_path))
    assert C.load().fbcorr_rtcg_check(C.I64_3(128, 140, 8), C.I64_4(64, 9, 9, 8), C.epilogue((0.0, 1.0)), b"f32tc", None,
                                      0) == 0
    names, text = _kernels(tmp_path)
    assert names == {"fbc_f32tc_", "fbc_f32dw_"} and "fl0_e1_m0" in text and "fl1_e0_m1" in text


def test_batch_rtcg_check_compiles_the_tensor_core_kernels(tmp_path, monkeypatch):
    monkeypatch.setenv("FBCORR_DUMP_DIR", str(tmp_path))
    shapes = [(200, 210, 8, 64, 7, 7), (12, 12, 3, 5, 2, 2), (200, 210, 8, 64, 7, 7)]
    ins = (ctypes.c_int64 * 9)(*[v for s in shapes for v in s[:3]])
    fls = (ctypes.c_int64 * 12)(*[v for s in shapes for v in (s[3], s[4], s[5], s[2])])
    assert C.load().fbcorr_batch_rtcg_check(3, ins, fls, C.epilogue(None), None, 0) == 0
    names, text = _kernels(tmp_path)
    assert names == {"fbc_f32tc_", "fbc_batch("} and len(list(tmp_path.iterdir())) == 2
    assert text.count("FbcV0") and text.count("FbcV1")     # the persistent kernel holds every image


@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("which", ["forward", "dx", "dw"])
def test_the_accuracy_question_tells_the_three_way_split_from_less(which, positive):
    """The bound that the GPU tests put on the kernels' errors holds for the six products
    that they keep and fails for a kernel that leaves the third order out (of random
    signs: in sums of one sign that order averages out)."""
    rng = np.random.default_rng(11)
    for case in {"forward": f32split.FORWARD, "dx": f32split.GRADIENT, "dw": f32split.BANK}[which]:
        x, w, g = f32split.layer(rng, case if which == "dw" else case[0], positive)
        op, a, b = {"forward": (oracle.fwd, x, w),
                    "dx": (lambda u, v: oracle.bwd_input(u, v, x.shape), g, w),
                    "dw": (lambda u, v: oracle.bwd_filt(u, v, w.shape), x, g)}[which]
        ref = op(a, b)
        assert f32split.rel2(f32split.six_products(op, a, b), ref) <= 2.0 ** -24
        if not positive:
            assert f32split.rel2(f32split.six_products(op, a, b, 2), ref) > f32split.NORMWISE


def test_left_out_products_are_below_two_to_the_minus_24():
    """x2 w3 and x3 w2 are below 2^-25 of |x w| each, and all three products together
    below 2^-24 (not 2^-26: x = w = 1.0038986 leaves out 2^-24.01)."""
    rng = np.random.default_rng(12)
    x = np.concatenate([rng.uniform(1, 2, 200000).astype(np.float32), np.float32([1.0038986, 1.00390619, 1.0039])])
    w = np.concatenate([rng.uniform(1, 2, 200000).astype(np.float32), np.float32([1.0038986, 1.00390619, 1.0039])])
    (_, x2, x3), (_, w2, w3) = ([p.astype(np.float64) for p in f32split.split3(v)] for v in (x, w))
    xw = x.astype(np.float64) * w
    assert np.all(np.abs(x2 * w3) < 2.0 ** -25 * xw) and np.all(np.abs(x3 * w2) < 2.0 ** -25 * xw)
    left = np.abs(x2 * w3 + x3 * w2 + x3 * w3)
    assert np.all(left < 2.0 ** -24 * xw) and left[-3] > 2.0 ** -24.1 * xw[-3]


@pytest.mark.parametrize("dtype,shape", [(0, (128, 140, 8, 64, 9, 9)), (1, (512, 512, 4, 32, 13, 13)),
                                         (2, (512, 512, 4, 32, 13, 13))])
def test_snippet_check_compiles_the_packed_kernels(dtype, shape, tmp_path, monkeypatch):
    monkeypatch.setenv("FBCORR_DUMP_DIR", str(tmp_path))
    H, W, D, N, fh, fw = shape
    assert C.load().fbcorr_snippet_check(C.I64_3(H, W, D), C.I64_4(N, fh, fw, D), dtype, b"y > 0.f ? y : lo * y", None,
                                         0) == 0
    text = "".join(f.read_text() for f in tmp_path.iterdir())
    assert len(list(tmp_path.iterdir())) == 2 and ("fbc_f32tc_f", "fbc_tcpack1_f", "fbc_tcpack2_f")[dtype] in text
