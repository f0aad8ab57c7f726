"""The packed tensor-core kernel of the BF16 modes against the modes' own kernel.

Both sum the same BF16 products in FP32; the packed kernel truncates at most 32 steps
before it adds up in registers, the other one every step of the sum: their difference
is at most (steps of both) * 2^-23 * sum |x| |w|.
"""
import numpy as np
import pytest

import oracle
from paper_0911_3456_gb300 import inputs
from helpers import dev, host, torch_cuda

pytestmark = pytest.mark.gpu

CASES = [
    ((20, 37, 1, 5, 3, 4), "tcpack:nt=16,r=1,gc=8,jt=4,ru=2"),
    ((33, 40, 4, 4, 8, 8), "tcpack:nt=32,r=8,gc=8,jt=8,ru=4"),
    ((25, 31, 5, 6, 3, 3), "tcpack:nt=16,r=1,gc=8,jt=3,ru=3"),
    ((60, 90, 8, 16, 9, 9), "tcpack:nt=64,r=4,gc=8,jt=9,ru=3"),
    ((31, 49, 24, 96, 7, 5), "tcpack:nt=96,r=1,gc=8,jt=5,ru=3"),
    ((18, 29, 20, 33, 2, 6), "tcpack:nt=48,r=1,gc=8,jt=4,ru=2"),
    ((60, 70, 64, 32, 5, 5), "tcpack:nt=96,r=3,gc=32,jt=5,ru=1"),
    ((15, 300, 32, 180, 3, 5), "tcpack:nt=96,r=1,gc=16,jt=5,ru=2"),
]


@pytest.mark.parametrize("mode", ["bf16", "bf16x3"])
@pytest.mark.parametrize("shape,spec", CASES)
def test_packed_against_the_modes_own_kernel(shape, spec, mode):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    for kind in ("int", "real"):
        wl = inputs.random_case(8100, *shape, kind=kind)
        x, w = dev(wl.x, torch), dev(wl.w, torch)
        p = Plan(wl.x.shape, wl.w.shape, mode, (-30.0, 30.0))
        p.set_variant(p.candidates()[0])
        ref = host(p.forward(x, w))
        p.set_variant(spec)
        assert p.info()["fwd"]["spec"] == spec
        y = host(p.forward(x, w))
        assert p.device_status() == 0
        if kind == "int":
            assert np.array_equal(y, np.clip(oracle.fwd(wl.x, wl.w), -30, 30)) and np.array_equal(y, ref)
        else:
            steps = 3 * shape[4] * shape[5] * ((shape[2] + 15) // 16)
            mag = oracle.fwd(np.abs(wl.x), np.abs(wl.w))
            assert np.all(np.abs(y - ref) <= (2 * steps + 8) * 2.0 ** -23 * mag)


@pytest.mark.parametrize("mode", ["bf16", "bf16x3"])
def test_packed_non_finite_values(mode):
    """Infinities and NaN reach the outputs that read them and no others (a folded row or
    a padded tap multiplies them by zero)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(8200, 24, 30, 8, 12, 5, 3)
    x = wl.x.copy()
    x[3, 4, 0], x[9, 20, 1], x[23, 29, 7] = np.inf, np.nan, -np.inf
    p = Plan(x.shape, wl.w.shape, mode)
    out = []
    for spec in (p.candidates()[0], "tcpack:nt=48,r=4,gc=8,jt=3,ru=2"):
        p.set_variant(spec)
        out.append(p.forward(dev(x, torch), dev(wl.w, torch)).cpu().numpy())
    a, b = out
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
    assert np.array_equal(a[np.isinf(a)], b[np.isinf(b)])


@pytest.mark.parametrize("mode", ["bf16", "bf16x3"])
@pytest.mark.parametrize("shape", [
    (140, 160, 16, 256, 2, 2),    # one 256-wide filter tile, more pixel tiles than SMs
    (141, 157, 20, 256, 3, 6),    # the same, ragged: rows no multiple of 32 pixels, taps past a stage
    (100, 160, 16, 256, 2, 2),    # fewer pixel tiles than SMs
    (130, 133, 16, 257, 2, 3),    # two filter tiles
    (20, 41, 33, 96, 3, 7),       # rows too deep for register conversion
])
def test_untuned_configuration_is_exact_on_integers(shape, mode, monkeypatch):
    """An untuned plan starts from the first candidate; integer sums are exact in it."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    monkeypatch.setenv("FBCORR_TCPACK", "0")
    wl = inputs.random_case(8300, *shape, kind="int")
    p = Plan(wl.x.shape, wl.w.shape, mode)
    assert p.info()["fwd"]["spec"] == p.candidates()[0]
    y = host(p.forward(dev(wl.x, torch), dev(wl.w, torch)))
    assert p.device_status() == 0
    assert np.array_equal(y, oracle.fwd(wl.x, wl.w))
