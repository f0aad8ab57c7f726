"""FP32 on the tensor cores (three-way BF16 split) against the FP64 oracle.

Tolerance, derived from the arithmetic: a chunk of at most 16 steps truncates its
FP32 accumulator by at most one unit (2^-23) of the magnitude summed so far at each
step, the chunk sums are added with ordinary rounding, and the products left out are
below 2^-26: |error| <= (16 * 2^-23 + (chunks + 4) * 2^-24) * sum |x| |w|.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import f32split
import oracle
from paper_0911_3456_gb300 import inputs
from helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu

# (H, W, D, N, fh, fw), forced tile: every depth layout (packed 1, 2, 4 and 8
# channels, 16 and 32 per unit, odd depths), tap groups, folded rows with a ragged
# last fold, several slab rows per unit with a ragged last unit, one and several
# filter tiles, filters past the tile, pixel tiles with a ragged end, one pixel
CASES = [
    ((20, 37, 1, 5, 3, 4), "f32tc:nt=16,r=1,gc=8,jt=4,ru=2"),
    ((19, 30, 2, 9, 4, 5), "f32tc:nt=32,r=3,gc=8,jt=5,ru=4"),
    ((21, 33, 3, 7, 2, 3), "f32tc:nt=16,r=2,gc=8,jt=3,ru=1"),
    ((33, 40, 4, 4, 8, 8), "f32tc:nt=32,r=8,gc=8,jt=8,ru=4"),
    ((25, 31, 5, 6, 3, 3), "f32tc:nt=16,r=1,gc=8,jt=3,ru=3"),
    ((30, 47, 8, 16, 9, 9), "f32tc:nt=64,r=4,gc=8,jt=5,ru=2"),
    ((17, 140, 12, 40, 5, 3), "f32tc:nt=48,r=1,gc=16,jt=3,ru=3"),
    ((18, 29, 20, 33, 2, 6), "f32tc:nt=48,r=1,gc=8,jt=4,ru=2"),
    ((23, 26, 16, 64, 7, 7), "f32tc:nt=64,r=1,gc=16,jt=7,ru=2"),
    ((15, 300, 32, 90, 3, 5), "f32tc:nt=48,r=1,gc=32,jt=5,ru=1"),
    ((16, 21, 33, 17, 5, 11), "f32tc:nt=32,r=1,gc=16,jt=6,ru=1"),
    ((12, 13, 64, 160, 1, 1), "f32tc:nt=80,r=1,gc=32,jt=1,ru=1"),
    ((6, 7, 8, 3, 6, 7), "f32tc:nt=16,r=1,gc=8,jt=7,ru=3"),
    ((4, 1, 4, 1, 2, 1), "f32tc:nt=16,r=3,gc=8,jt=1,ru=1"),
]


def _within(got, ref, mag, chunks):
    assert np.all(np.abs(got - ref) <= (16 * 2.0 ** -23 + (chunks + 4) * 2.0 ** -24) * mag + 1e-30)


@pytest.mark.parametrize("shape,spec", CASES)
def test_forward_against_oracle_and_integers(shape, spec):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    for kind in ("real", "int"):
        wl = inputs.random_case(7100, *shape, kind=kind)
        p = Plan(wl.x.shape, wl.w.shape)
        p.set_variant(spec)
        assert p.info()["fwd"]["spec"] == spec
        y = host(p.forward(dev(wl.x, torch), dev(wl.w, torch)))
        assert p.device_status() == 0
        ref = oracle.fwd(wl.x, wl.w)
        if kind == "int":
            assert np.array_equal(y, ref)
        else:
            _within(y, ref, oracle.fwd(np.abs(wl.x), np.abs(wl.w)), shape[2] * shape[4] * shape[5])


@pytest.mark.parametrize("clamp", [None, (-0.5, 0.5)])
@pytest.mark.parametrize("shape,spec", [
    ((20, 23, 16, 64, 7, 7), "f32tc:nt=64,r=4,gc=32,jt=7,ru=1"),
    ((19, 26, 12, 40, 5, 3), "f32tc:nt=48,r=3,gc=8,jt=3,ru=4"),
    ((24, 31, 5, 7, 3, 4), "f32tc:nt=16,r=1,gc=8,jt=4,ru=2"),
    ((17, 40, 33, 3, 2, 5), "f32tc:nt=48,r=1,gc=8,jt=3,ru=1"),
])
def test_dx_against_oracle(shape, spec, clamp, monkeypatch):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_DX_VARIANT", spec)
    wl = inputs.random_case(7200, *shape, with_g=True)
    p = Plan(wl.x.shape, wl.w.shape, "f32", clamp)
    y64 = oracle.fwd(wl.x, wl.w, epilogue=clamp)
    y = y64.astype(np.float32)
    dx, _ = p.backward(dev(wl.x, torch), dev(wl.w, torch), dev(wl.g, torch), dev(y, torch), need_dw=False)
    assert p.info()["dx"]["spec"] == spec
    assert p.device_status() == 0
    ref = oracle.bwd_input(wl.g, wl.w, wl.x.shape, y=y.astype(np.float64), epilogue=clamp)
    mag = oracle.bwd_input(np.abs(wl.g), np.abs(wl.w), wl.x.shape)
    _within(host(dx), ref, mag, shape[3] * shape[4] * shape[5])


# one and several filter tiles, 32- and 64-row blocks, one and two planes of x per CTA
# with a half-empty and an empty last plane, odd and even filter widths, two tap
# groups, ragged last chunks, images smaller than a chunk, a single column
DW_SHAPES = [(30, 41, 16, 64, 7, 7), (19, 26, 12, 40, 5, 3), (24, 31, 4, 8, 3, 4), (17, 40, 24, 132, 2, 5),
             (40, 33, 8, 20, 9, 9), (25, 29, 32, 68, 4, 13), (21, 60, 4, 36, 2, 19), (9, 11, 20, 4, 3, 1),
             (5, 1, 8, 64, 2, 1)]


@pytest.mark.parametrize("clamp", [None, (-0.5, 0.5)])
@pytest.mark.parametrize("shape", DW_SHAPES)
def test_dw_against_oracle_and_integers(shape, clamp, monkeypatch):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_F32TC", "force")
    for kind in ("real", "int"):
        wl = inputs.random_case(7700, *shape, kind=kind, with_g=True)
        p = Plan(wl.x.shape, wl.w.shape, "f32", clamp)
        y = oracle.fwd(wl.x, wl.w, epilogue=clamp).astype(np.float32)
        args = (dev(wl.x, torch), dev(wl.w, torch), dev(wl.g, torch), dev(y, torch))
        dw = p.backward(*args, need_dx=False)[1]
        assert "f32tc" in p.info()["dw"] and p.device_status() == 0
        assert torch.equal(dw, p.backward(*args)[1])          # with dL/dx beside it, run to run
        ref = oracle.bwd_filt(wl.x, wl.g, wl.w.shape, y=y.astype(np.float64), epilogue=clamp)
        if kind == "int":
            assert np.array_equal(host(dw), ref)
        else:
            mag = oracle.bwd_filt(np.abs(wl.x), np.abs(wl.g), wl.w.shape)
            _within(host(dw), ref, mag, shape[0] * shape[1] // 96 + 64)


@pytest.mark.parametrize("what", ["inf", "nan", "tiny_g", "tiny_x"])
def test_dw_values_outside_the_split(what, monkeypatch):
    """They come from the FMA kernel, as a plan without the tensor-core kernel computes them."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7800, 30, 41, 16, 64, 5, 5, with_g=True)
    x, g = wl.x.copy(), wl.g.copy()
    if what == "inf":
        x[7, 40, 3] = np.inf            # a column that the last output columns alone read
    elif what == "nan":
        g[3, 4, 5] = np.nan
    elif what == "tiny_g":
        g *= np.float32(1e-34)
    else:
        x[2, 3, 4] = 1e-33
    out = []
    for sw in ("force", "0"):
        monkeypatch.setenv("FBCORR_F32TC", sw)
        p = Plan(x.shape, wl.w.shape)
        out.append(p.backward(dev(x, torch), dev(wl.w, torch), dev(g, torch), need_dx=False)[1].cpu().numpy())
        assert ("f32tc" in p.info()["dw"]) == (sw == "force")
    assert np.array_equal(out[0], out[1], equal_nan=True)


def _special(shape):
    """Inputs the BF16 split cannot carry: non-finite, at the range's ends, denormal."""
    wl = inputs.random_case(7300, *shape)
    x = wl.x.copy()
    x[3, 4, 0] = np.inf
    x[9, 20, 1] = np.nan
    x[14, 7, 0] = -3.3e38
    x[18, 25, 2] = 1e-39
    return x, wl.w


def test_values_outside_the_split_match_the_fma_kernel():
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    x, w = _special((24, 30, 8, 20, 3, 3))
    xd, wd = dev(x, torch), dev(w, torch)
    p = Plan(x.shape, w.shape)
    p.set_variant("f32tc:nt=32,r=1,gc=8,jt=3,ru=3")
    y = p.forward(xd, wd).cpu().numpy()
    p.set_variant("default")
    ref = p.forward(xd, wd).cpu().numpy()
    assert np.array_equal(np.isnan(y), np.isnan(ref))
    assert np.array_equal(np.isinf(y), np.isinf(ref)) and np.array_equal(y[np.isinf(y)], ref[np.isinf(ref)])
    fin = np.isfinite(ref)
    with np.errstate(all="ignore"):
        exact, mag = oracle.fwd(x, w), oracle.fwd(np.abs(x), np.abs(w))
    _within(y[fin].astype(np.float64), exact[fin], mag[fin], 72)


@pytest.mark.parametrize("scale_x,scale_w", [(1e-33, 1.0), (1.0, 1e-34), (1e-38, 1e20), (1e19, 1e18)])
def test_extreme_scales_keep_fp32_accuracy(scale_x, scale_w):
    """Tiny images and banks (the third part of the split would underflow) and large ones."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7400, 20, 40, 8, 18, 3, 3)
    x, w = (wl.x * np.float32(scale_x)), (wl.w * np.float32(scale_w))
    p = Plan(x.shape, w.shape)
    p.set_variant("f32tc:nt=32,r=1,gc=8,jt=3,ru=3")
    y = host(p.forward(dev(x, torch), dev(w, torch)))
    ref = oracle.fwd(x, w)
    mag = oracle.fwd(np.abs(x), np.abs(w))
    assert np.all(np.abs(y - ref) <= 2.0 ** -18 * mag + 1e-44)


def test_scratch_too_small_runs_the_fma_kernel():
    """Any workspace is accepted: none, or less than the kernel wants, gives the FMA result."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7500, 40, 50, 8, 32, 5, 5)
    x, w = dev(wl.x, torch), dev(wl.w, torch)
    p = Plan(wl.x.shape, wl.w.shape)
    p.set_variant("f32tc:nt=32,r=1,gc=8,jt=5,ru=2")
    y3 = p.forward(x, w)
    small = p.forward(x, w, ws=torch.empty(64, dtype=torch.uint8, device="cuda"))
    assert p.ws_fwd == 0
    ref = oracle.fwd(wl.x, wl.w)
    scale = np.abs(ref).max()
    assert np.abs(host(y3) - ref).max() <= 1e-6 * scale and np.abs(host(small) - ref).max() <= 1e-6 * scale
    from paper_0911_3456_gb300 import _capi as C
    import ctypes
    y = torch.empty_like(small)
    C.call("fbcorr_forward", p.handle, *[ctypes.c_void_p(t.data_ptr()) for t in (x, w, y)], None, 0, None)
    torch.cuda.synchronize()
    assert torch.equal(y, small)


def test_streams_and_capture():
    """Overlapping calls of one plan on two streams, and a call captured in a graph."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7600, 64, 80, 16, 48, 5, 5)
    p = Plan(wl.x.shape, wl.w.shape)
    p.set_variant("f32tc:nt=48,r=1,gc=16,jt=5,ru=2")
    x, w = dev(wl.x, torch), dev(wl.w, torch)
    x2, w2 = x * 2, w * 3
    y = p.forward(x, w)
    y2 = p.forward(x2, w2)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(5):
        a = p.forward(x, w, torch.empty_like(y), stream=s1)
        b = p.forward(x2, w2, torch.empty_like(y), stream=s2)
        torch.cuda.synchronize()
        assert torch.equal(a, y) and torch.equal(b, y2)
    g = torch.cuda.CUDAGraph()
    out = torch.empty_like(y)
    with torch.cuda.graph(g):
        p.forward(x, w, out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, y)
    x.copy_(x2)
    w.copy_(w2)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, y2)


def test_no_memory_for_the_scratch_runs_the_fma_kernels(monkeypatch):
    """The scratch is optional: where the device has no memory for it, the calls give
    what the FMA kernels give, bit for bit."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7190, 160, 170, 16, 64, 7, 7)
    x, w = dev(wl.x, torch), dev(wl.w, torch)
    p = Plan(wl.x.shape, wl.w.shape)
    g = torch.rand(p.out_shape, device="cuda") - 0.5
    assert p.info()["fwd"]["spec"].startswith("f32tc:") and p._scratch_size(True) > p.ws_bwd
    small = torch.empty(16, dtype=torch.uint8, device="cuda")   # too small for any scratch
    y0 = p.forward(x, w, ws=small)
    dx0, dw0 = p.backward(x, w, g, ws=p.workspace(p.ws_bwd, x.device))
    empty = torch.empty

    def full(*size, dtype=None, **kw):
        if dtype is torch.uint8 and size[0] != p.ws_bwd:
            raise torch.cuda.OutOfMemoryError("no memory")
        return empty(*size, dtype=dtype, **kw)

    monkeypatch.setattr(torch, "empty", full)
    y1 = p.forward(x, w)
    dx1, dw1 = p.backward(x, w, g)
    assert torch.equal(y0, y1) and torch.equal(dx0, dx1) and torch.equal(dw0, dw1)
    dx2, none = p.backward(x, w, g, need_dw=False)
    assert none is None and torch.equal(dx0, dx2)


@pytest.mark.parametrize("clamp", [None, (-20.0, 25.0)])
@pytest.mark.parametrize("where", ["g", "w"])
def test_dx_non_finite_values_against_oracle(where, clamp, monkeypatch):
    """Infinities and NaN in the gradient or the filters reach the pixels of dL/dx that
    read them, the border's (where a filter value meets no gradient) as elsewhere, and
    the finite values are exact on integers."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_DX_VARIANT", "f32tc:nt=32,r=1,gc=8,jt=3,ru=2")
    wl = inputs.random_case(7195, 30, 41, 8, 24, 5, 3, kind="int", with_g=True)
    p = Plan(wl.x.shape, wl.w.shape, "f32", clamp)
    y = p.forward(dev(wl.x, torch), dev(wl.w, torch))
    g, w = wl.g.copy(), wl.w.copy()
    if where == "g":
        g[0, 0, 0], g[12, 20, 7], g[25, 38, 23] = np.inf, np.nan, -np.inf
    else:
        w[3, 2, 1, 0], w[9, 0, 2, 5], w[20, 4, 0, 7] = np.inf, np.nan, -np.inf
    dx = p.backward(dev(wl.x, torch), dev(w, torch), dev(g, torch), y=y, need_dw=False)[0].cpu().numpy()
    assert p.info()["dx"]["spec"].startswith("f32tc") and p.device_status() == 0
    with np.errstate(all="ignore"):
        ref = oracle.bwd_input(g, w, wl.x.shape, y=host(y), epilogue=clamp)
    assert np.array_equal(dx, ref, equal_nan=True)


def _us(torch, f, calls=8, rounds=6):
    """Least time of a call among others, from a graph: without the host's part."""
    f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(calls):
            f()
    best = float("inf")
    for _ in range(rounds + 1):            # the first round warms up
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / calls * 1e3)
    return best


@pytest.mark.parametrize("shape", [(256, 256, 16, 64, 7, 7), (512, 700, 4, 4, 8, 8)])
def test_tiny_values_do_not_slow_the_calls(shape):
    """Denormal and tiny weights, pixels and gradients split like any other value: a call
    with them takes what the call without them takes (it took 10 to 1000 times that)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    H, W, D, N, fh, fw = shape
    gen = torch.Generator(device="cuda").manual_seed(7900)
    x = torch.rand((H, W, D), generator=gen, device="cuda") - 0.5
    w = torch.randn((N, fh, fw, D), generator=gen, device="cuda")
    p = Plan(x.shape, w.shape)
    g = torch.randn(p.out_shape, generator=gen, device="cuda")
    x1, w1, g1 = x.clone(), w.clone(), g.clone()
    x1.view(-1)[::997] = 1e-33
    w1[N // 2, 1, 1, 1] = -1e-38
    g1.view(-1)[::997] = 1e-40
    plain = _us(torch, lambda: p.forward(x, w)), _us(torch, lambda: p.backward(x, w, g, need_dw=False))
    assert p.info()["fwd"]["kind"] == "f32tc" and p.info()["dx"]["kind"] == "f32tc"
    for a, b in ((x1, w), (x, w1)):
        assert _us(torch, lambda: p.forward(a, b)) <= 1.5 * plain[0]
    for b, c in ((w1, g), (w, g1)):
        assert _us(torch, lambda: p.backward(x, b, c, need_dw=False)) <= 1.5 * plain[1]


@pytest.mark.parametrize("ex,ew", [(-70, -70), (-66, -73), (-100, -40), (-126, -14), (-140, 20), (30, -140)])
def test_small_values_and_products_keep_fp32_accuracy(ex, ew, monkeypatch):
    """Operands down to the denormal ones, and results near the end of the range: the
    error is the file's bound with the kernel's one chunk, and one rounding to a
    multiple of 2^-149 (derived: the sums are held 2^32 times larger)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_DX_VARIANT", "f32tc:nt=16,r=1,gc=16,jt=3,ru=3")
    wl = inputs.random_case(7950, 20, 40, 8, 16, 3, 3, with_g=True)
    x, w, g = wl.x * np.float32(2.0 ** ex), wl.w * np.float32(2.0 ** ew), wl.g * np.float32(2.0 ** ex)
    p = Plan(x.shape, w.shape)
    p.set_variant("f32tc:nt=32,r=1,gc=8,jt=3,ru=3")
    y = host(p.forward(dev(x, torch), dev(w, torch)))
    dx = host(p.backward(dev(x, torch), dev(w, torch), dev(g, torch), need_dw=False)[0])
    assert p.info()["dx"]["spec"].startswith("f32tc")
    for got, ref, mag in ((y, oracle.fwd(x, w), oracle.fwd(np.abs(x), np.abs(w))),
                          (dx, oracle.bwd_input(g, w, x.shape), oracle.bwd_input(np.abs(g), np.abs(w), x.shape))):
        assert np.all(np.abs(got - ref) <= (16 * 2.0 ** -23 + 5 * 2.0 ** -24) * mag + 2.0 ** -149)


@pytest.mark.parametrize("ex,eg", [(-70, -70), (-66, -66), (-95, -40), (60, 60)])
def test_dw_small_products_keep_fp32_accuracy(ex, eg, monkeypatch):
    """dL/dw near the end of the range (every value of the split's range, sums near
    2^-130): the bound of one chunk per 96 pixels and partial sum, and one rounding to a
    multiple of 2^-149 for each of the at most 40 partial sums and their total; and
    sums that the kernel holds 2^32 times larger than FP32 could: from the FMA kernel."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_F32TC", "force")
    wl = inputs.random_case(7960, 30, 41, 16, 64, 5, 5, with_g=True)
    least = np.float32(2.0 ** -4)              # no value below the split's range
    x = np.where(np.abs(wl.x) < least, least, wl.x) * np.float32(2.0 ** ex)
    g = np.where(np.abs(wl.g) < least, least, wl.g) * np.float32(2.0 ** eg)
    p = Plan(x.shape, wl.w.shape)
    dw = host(p.backward(dev(x, torch), dev(wl.w, torch), dev(g, torch), need_dx=False)[1])
    assert "f32tc" in p.info()["dw"] and p.device_status() == 0
    ref, mag = oracle.bwd_filt(x, g, wl.w.shape), oracle.bwd_filt(np.abs(x), np.abs(g), wl.w.shape)
    assert np.all(np.abs(dw - ref) <= (16 * 2.0 ** -23 + 64 * 2.0 ** -24) * mag + 41 * 2.0 ** -150)


def _spoiled(t):
    """Integers with a NaN, an infinity and a value whose sums leave the split's range."""
    t = t.copy()
    f = t.reshape(-1)
    f[f.size // 3], f[f.size // 2], f[2 * f.size // 3] = np.nan, -np.inf, 2.0 ** 100
    return t


def _same_as_oracle(got, ref, mag, terms):
    """Non-finite values alike, integers equal, and sums with 2^100 in them within the
    rounding of one FMA per term."""
    fin = np.isfinite(ref)
    assert np.array_equal(got[~fin], ref[~fin], equal_nan=True)
    small = fin & (mag < 2.0 ** 24)
    assert np.array_equal(got[small], ref[small])
    assert np.all(np.abs(got[fin] - ref[fin]) <= (terms + 4) * 2.0 ** -24 * mag[fin])


@pytest.mark.parametrize("where", ["x", "w"])
@pytest.mark.parametrize("shape,spec", CASES)
def test_recomputed_outputs_in_every_layout(shape, spec, where):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7970, *shape, kind="int")
    x, w = (_spoiled(wl.x), wl.w) if where == "x" else (wl.x, _spoiled(wl.w))
    p = Plan(x.shape, w.shape)
    p.set_variant(spec)
    y = host(p.forward(dev(x, torch), dev(w, torch)))
    assert p.device_status() == 0
    with np.errstate(all="ignore"):
        _same_as_oracle(y, oracle.fwd(x, w), oracle.fwd(np.abs(x), np.abs(w)), shape[2] * shape[4] * shape[5])


@pytest.mark.parametrize("clamp", [None, (-20.5, 20.5)])
@pytest.mark.parametrize("where", ["g", "w"])
@pytest.mark.parametrize("shape,spec", [
    ((20, 23, 16, 64, 7, 7), "f32tc:nt=64,r=4,gc=32,jt=7,ru=1"),
    ((19, 26, 12, 40, 5, 3), "f32tc:nt=48,r=3,gc=8,jt=3,ru=4"),
    ((24, 31, 5, 7, 3, 4), "f32tc:nt=16,r=1,gc=8,jt=4,ru=2"),
    ((17, 40, 33, 3, 2, 5), "f32tc:nt=48,r=1,gc=8,jt=3,ru=1"),
    ((22, 31, 6, 12, 3, 3), "f32tc:nt=32,r=5,gc=8,jt=3,ru=2"),
])
def test_recomputed_gradients_in_every_layout(shape, spec, where, clamp, monkeypatch):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_DX_VARIANT", spec)
    wl = inputs.random_case(7980, *shape, kind="int", with_g=True)
    g, w = (_spoiled(wl.g), wl.w) if where == "g" else (wl.g, _spoiled(wl.w))
    p = Plan(wl.x.shape, w.shape, "f32", clamp)
    y = oracle.fwd(wl.x, wl.w, epilogue=clamp).astype(np.float32)
    dx = host(p.backward(dev(wl.x, torch), dev(w, torch), dev(g, torch), dev(y, torch), need_dw=False)[0])
    assert p.info()["dx"]["spec"] == spec and p.device_status() == 0
    with np.errstate(all="ignore"):
        ref = oracle.bwd_input(g, w, wl.x.shape, y=y.astype(np.float64), epilogue=clamp)
        mag = oracle.bwd_input(np.abs(g), np.abs(w), wl.x.shape, y=y.astype(np.float64), epilogue=clamp)
    _same_as_oracle(dx, ref, mag, shape[3] * shape[4] * shape[5])


def test_more_recomputed_groups_than_a_block_notes():
    """NaN in most groups of pixels: past its list a block computes whole items again."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(7985, 702, 900, 4, 16, 2, 2, kind="int")
    x = wl.x.copy()
    x.reshape(-1)[::97] = np.nan
    p = Plan(x.shape, wl.w.shape)
    p.set_variant("f32tc:nt=16,r=1,gc=8,jt=2,ru=2")
    y = host(p.forward(dev(x, torch), dev(wl.w, torch)))
    assert p.device_status() == 0
    assert np.array_equal(y, oracle.fwd(x, wl.w), equal_nan=True)


@pytest.mark.parametrize("shape", [(256, 256, 16, 64, 7, 7), (512, 700, 4, 4, 8, 8)])
def test_non_finite_values_cost_no_more_than_a_few_fma_kernels(shape):
    """A NaN weight, one NaN pixel or one NaN gradient, and NaN everywhere: at most four
    times what the FMA kernels take for the whole call (it was 20 to 1000 times)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    H, W, D, N, fh, fw = shape
    gen = torch.Generator(device="cuda").manual_seed(7990)
    x = torch.rand((H, W, D), generator=gen, device="cuda") - 0.5
    w = torch.randn((N, fh, fw, D), generator=gen, device="cuda")
    p = Plan(x.shape, w.shape)
    g = torch.randn(p.out_shape, generator=gen, device="cuda")
    small = torch.empty(16, dtype=torch.uint8, device="cuda")     # no scratch: the FMA kernels
    x1, x2, w1, g1, g2 = x.clone(), x.clone(), w.clone(), g.clone(), g.clone()
    x1[H // 2, W // 3, 1] = w1[N // 2, 1, 1, 1] = g1[H // 2, W // 3, 1] = float("nan")
    x2.view(-1)[::997] = g2.view(-1)[::997] = float("nan")
    fma = (_us(torch, lambda: p.forward(x, w, ws=small)), _us(torch, lambda: p.backward(x, w, g, need_dw=False, ws=small)))
    for a, b in ((x1, w), (x2, w), (x, w1)):
        assert _us(torch, lambda: p.forward(a, b)) <= 4 * fma[0]
    for b, c in ((w1, g), (w, g1), (w, g2)):
        assert _us(torch, lambda: p.backward(x, b, c, need_dw=False)) <= 4 * fma[1]


def test_calls_without_scratch_run_the_tuned_fma_kernels(tmp_path, monkeypatch):
    """Where the tuner picks the tensor-core kernel, the plan, and plans made from the
    cache, keep the FMA kernel that it measured fastest for calls without scratch."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_CACHE_DIR", str(tmp_path))
    monkeypatch.setenv("FBCORR_TUNE_TOPK", "2")
    wl = inputs.random_case(7995, 200, 230, 8, 64, 7, 7, with_g=True)
    x, w, g = dev(wl.x, torch), dev(wl.w, torch), dev(wl.g, torch)
    p = Plan(wl.x.shape, wl.w.shape)
    p.autotune()
    p.backward(x, w, g, need_dw=False)
    assert p.info()["fwd"]["kind"] == "f32tc" and p.info()["dx"]["kind"] == "f32tc"
    path = tmp_path / "tune.tsv"
    saved = dict(line.split("\t") for line in path.read_text().splitlines())
    fwd, dx = (next(k for k in saved if k.endswith("|fma") and f"{what}|x" in k) for what in ("fwd", "dx"))
    assert p.info()["fwd"]["fma"] == saved[fwd] and p.info()["dx"]["fma"] == saved[dx]
    # other kernels in the cache are the ones that run: their bits, without scratch
    small = torch.empty(16, dtype=torch.uint8, device="cuda")
    for fma in ({fwd: "direct:tr=2,tf=4,wr=4,wf=2,cc=0,pk=1", dx: "direct:tr=2,tf=4,wr=2,wf=2,cc=16,pk=1"},
                {fwd: "default", dx: "default"}):
        path.write_text("".join(f"{k}\t{fma.get(k, v)}\n" for k, v in saved.items()))
        q = Plan(wl.x.shape, wl.w.shape)
        assert q.info()["fwd"]["source"] == "cache" and q.info()["fwd"]["kind"] == "f32tc"
        y, gx = q.forward(x, w, ws=small), q.backward(x, w, g, need_dw=False, ws=small)[0]
        assert q.info()["fwd"]["fma"] == fma[fwd] and q.info()["dx"]["fma"] == fma[dx]
        monkeypatch.setenv("FBCORR_DX_VARIANT", fma[dx])
        r = Plan(wl.x.shape, wl.w.shape)
        r.set_variant(fma[fwd])
        assert torch.equal(y, r.forward(x, w)) and torch.equal(gx, r.backward(x, w, g, need_dw=False)[0])
        monkeypatch.delenv("FBCORR_DX_VARIANT")


def _three_passes(torch, which, x, w, g, spec, monkeypatch):
    """The pass on the tensor cores, the same on the FMA kernel, and the oracle's."""
    from paper_0911_3456_gb300.api import Plan
    xd, wd, gd = dev(x, torch), dev(w, torch), dev(g, torch)
    if which == "forward":
        p = Plan(x.shape, w.shape)
        p.set_variant(spec)
        out = p.forward(xd, wd), p.forward(xd, wd, ws=torch.empty(16, dtype=torch.uint8, device="cuda"))
        ref = oracle.fwd(x, w)
    elif which == "dx":
        monkeypatch.setenv("FBCORR_DX_VARIANT", spec)
        p = Plan(x.shape, w.shape)
        out = [p.backward(xd, wd, gd, need_dw=False, ws=ws)[0] for ws in
               (None, torch.empty(16, dtype=torch.uint8, device="cuda"))]
        assert p.info()["dx"]["spec"] == spec
        ref = oracle.bwd_input(g, w, x.shape)
    else:
        monkeypatch.setenv("FBCORR_F32TC", "force")
        p = Plan(x.shape, w.shape)
        out = [p.backward(xd, wd, gd, need_dx=False, ws=ws)[1] for ws in (None, p.workspace(p.ws_bwd, xd.device))]
        assert "f32tc" in p.info()["dw"]
        ref = oracle.bwd_filt(x, g, w.shape)
    assert p.device_status() == 0
    return host(out[0]), host(out[1]), ref


ACCURACY = ([("forward", s, t) for s, t in f32split.FORWARD] + [("dx", s, t) for s, t in f32split.GRADIENT] +
            [("dw", s, None) for s in f32split.BANK])


@pytest.mark.parametrize("positive", [False, True], ids=["signs", "positive"])
@pytest.mark.parametrize("which,shape,spec", ACCURACY)
def test_normwise_error_is_that_of_the_three_way_split(which, shape, spec, positive, monkeypatch):
    """A bound that a kernel without the third order breaks (tests/test_f32tc_cpu.py), and
    no more than twice the FMA kernel's error on the same values of random signs (sums of
    a few products may be exact there: one rounding of 2^-24 beside it).  In sums of one
    sign the truncations of a chunk do not average out."""
    torch = torch_cuda()
    x, w, g = f32split.layer(np.random.default_rng(8000), shape, positive)
    got, fma, ref = _three_passes(torch, which, x, w, g, spec, monkeypatch)
    err = f32split.rel2(got, ref)
    assert err <= f32split.NORMWISE
    if not positive:
        assert err <= 2 * f32split.rel2(fma, ref) + 2.0 ** -24


@pytest.mark.parametrize("which,shape,spec", ACCURACY)
def test_24_bit_values_pass_unchanged(which, shape, spec, monkeypatch):
    """Each sum holds one product with a power of two: every bit of the other factor comes
    through, whichever operand it is in."""
    torch = torch_cuda()
    rng = np.random.default_rng(8100)
    H, W, D, N, fh, fw = shape
    x, w, g = f32split.layer(rng, shape)

    def power():
        return np.float32(2.0 ** rng.integers(-3, 4)) * rng.choice(np.array([-1, 1], np.float32))

    def one_per_sum(op):
        """One operand with at most one non-zero value in each sum."""
        if op == "w_forward":                                  # one weight per filter
            v = np.zeros_like(w)
            for n in range(N):
                v[n, rng.integers(fh), rng.integers(fw), rng.integers(D)] = power()
        elif op == "x_forward":                                # pixels a filter apart
            v = np.zeros_like(x)
            for i in range(0, H, fh):
                for j in range(0, W, fw):
                    v[i, j, rng.integers(D)] = power()
        elif op == "w_dx":                                     # one weight per channel
            v = np.zeros_like(w)
            for d in range(D):
                v[rng.integers(N), rng.integers(fh), rng.integers(fw), d] = power()
        elif op == "g_dx":                                     # gradients a filter apart
            v = np.zeros_like(g)
            for i in range(0, g.shape[0], fh):
                for j in range(0, g.shape[1], fw):
                    v[i, j, rng.integers(N)] = power()
        elif op == "x_dw":                                     # one pixel per channel
            v = np.zeros_like(x)
            for d in range(D):
                v[rng.integers(H), rng.integers(W), d] = power()
        else:                                                  # one gradient per filter
            v = np.zeros_like(g)
            for n in range(N):
                v[rng.integers(g.shape[0]), rng.integers(g.shape[1]), n] = power()
        return v

    for op in {"forward": ("w_forward", "x_forward"), "dx": ("w_dx", "g_dx"), "dw": ("x_dw", "g_dw")}[which]:
        args = [one_per_sum(op) if op[0] == name else v for name, v in (("x", x), ("w", w), ("g", g))]
        got, _, ref = _three_passes(torch, which, *args, spec, monkeypatch)
        assert np.count_nonzero(ref) > 0
        # dL/dw adds first and third parts before the second: 25 bits where the first was rounded up
        assert np.all(np.abs(got - ref) <= 2.0 ** -23 * np.abs(ref)) if op == "x_dw" else np.array_equal(got, ref)


@pytest.mark.parametrize("shape", [(500, 341, 16, 64, 5, 4), (336, 396, 8, 64, 6, 2)])
def test_clamped_dw_is_not_slower_than_the_fma_kernel(shape):
    """Where a plan runs the masked dL/dw on the tensor cores (it took 1.2 and 1.5 times
    the FMA kernel's time here, with every mask value waited for as it was loaded)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    H, W, D, N, fh, fw = shape
    gen = torch.Generator(device="cuda").manual_seed(8200)
    x = torch.rand((H, W, D), generator=gen, device="cuda")
    w = torch.randn((N, fh, fw, D), generator=gen, device="cuda") / (fh * fw * D) ** 0.5
    p = Plan(x.shape, w.shape, clamp=(0.0, 1.0))
    y = p.forward(x, w)
    g = torch.randn(p.out_shape, generator=gen, device="cuda")
    p.backward(x, w, g, y, need_dx=False)
    assert "f32tc" in p.info()["dw"]
    fma = p.workspace(p.ws_bwd, x.device)
    assert (_us(torch, lambda: p.backward(x, w, g, y, need_dx=False)) <=
            _us(torch, lambda: p.backward(x, w, g, y, need_dx=False, ws=fma)))


def test_clamped_dx_is_not_slower_than_the_fma_kernel():
    """The same for dL/dx (it took 1.25 times the FMA kernel's time here)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    gen = torch.Generator(device="cuda").manual_seed(8300)
    x = torch.rand((2048, 2048, 4), generator=gen, device="cuda")
    w = torch.randn((4, 8, 8, 4), generator=gen, device="cuda") / 16
    p = Plan(x.shape, w.shape, clamp=(0.0, 1.0))
    y = p.forward(x, w)
    g = torch.randn(p.out_shape, generator=gen, device="cuda")
    p.backward(x, w, g, y, need_dw=False)
    assert p.info()["dx"]["kind"] == "f32tc"
    small = torch.empty(16, dtype=torch.uint8, device="cuda")
    assert (_us(torch, lambda: p.backward(x, w, g, y, need_dw=False)) <=
            _us(torch, lambda: p.backward(x, w, g, y, need_dw=False, ws=small)))


@pytest.mark.parametrize("dtype", ["f32", "bf16x3", "bf16"])
def test_candidates_are_what_the_tuner_times(dtype, tmp_path):
    """In a child process, whose log names every variant that is timed."""
    torch_cuda()
    code = ("import sys; from paper_0911_3456_gb300.api import Plan\n"
            f"p = Plan((70, 90, 8), (16, 5, 5, 8), {dtype!r}); c = p.candidates()\n"
            "for s in c:\n    if s.startswith(('f32tc', 'tcpack')): p.set_variant(s)\n"
            "print(\"\\n\".join(c)); p.autotune()")
    env = dict(os.environ, FBCORR_LOG="1", FBCORR_CACHE_DIR=str(tmp_path), FBCORR_TUNE_TOPK="3")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600, env=env,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr[-2000:]
    names = ("f32tc:", "tcpack:")
    listed = {s for s in r.stdout.split() if s.startswith(names)}
    # an FP32 plan tunes dL/dx as well, after the forward's pick is logged
    log = r.stderr.split("autotune fwd picked" if dtype == "f32" else "autotune picked")[0]
    timed = {word.rstrip(":") for line in log.splitlines() if "autotune" in line for word in line.split()
             if word.startswith(names)}
    assert listed and listed == timed
