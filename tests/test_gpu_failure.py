"""Failure detection on the GPU without faulting it: bounded waits that run
out report a status the host reads, code-generation failure falls back to the
prebuilt kernel, and a corrupt tuning cache is ignored."""
import os

import numpy as np
import pytest

import oracle
from helpers import dev, host, normwise_rel, torch_cuda
from paper_0911_3456_gb300 import inputs

pytestmark = pytest.mark.gpu


class _env:
    def __init__(self, **kv):
        self.kv = kv
        self.old = {}

    def __enter__(self):
        for k, v in self.kv.items():
            self.old[k] = os.environ.get(k)
            os.environ[k] = v

    def __exit__(self, *a):
        for k, v in self.old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


@pytest.mark.parametrize("spec,N", [(None, 32), ("tcgen05:na=2,nb=3,nt=256,bt=1,ew=8,fz=1,nr=0,cw=8,ts=1,sb=1", 32),
                                    ("tcgen05:na=2,nb=4,nt=256,bt=1,ew=4,fz=1,nr=0,cw=8,cg=2", 256)],
                         ids=["default", "staged_stores", "cta_pair"])
def test_dropped_copy_times_out_and_context_survives(spec, N):
    """FBCORR_FAULT=tcdrop makes the producer skip one copy that the MMA warp
    waits for -- an arrival that never comes.  Every wait is bounded (here
    50 ms): the kernel records FBCORR_ERR_TIMEOUT in host-mapped memory, drains
    its own copies and MMAs, frees TMEM and returns; the next plan on the same
    context computes correct results, with the default variant, with the
    staged-store epilogue, and with CTA pairs (both CTAs of a pair give up on
    their own bounded waits and meet at the closing cluster barrier)."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(3000, 20, 150, 16, N, 3, 3)
    x, w = dev(wl.x, torch), dev(wl.w, torch)
    with _env(FBCORR_FAULT="tcdrop", FBCORR_WAIT_MS="50"):
        bad = Plan(wl.x.shape, wl.w.shape, "bf16x3")
    if spec:
        bad.set_variant(spec)
    bad.forward(x, w)
    torch.cuda.synchronize()                    # the launch itself succeeds
    assert bad.device_status() == 9             # FBCORR_ERR_TIMEOUT
    assert bad.device_status(clear=True) == 9
    assert bad.device_status() == 0
    good = Plan(wl.x.shape, wl.w.shape, "bf16x3")
    y = host(good.forward(x, w))
    torch.cuda.synchronize()
    assert good.device_status() == 0
    assert normwise_rel(y, oracle.fwd(wl.x, wl.w)) <= 2e-5


def test_nvrtc_failure_falls_back_to_prebuilt_kernel(tmp_path):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(3100, 30, 41, 4, 6, 3, 3)
    with _env(FBCORR_FAULT="nvrtc,nocache", FBCORR_CACHE_DIR=str(tmp_path)):
        p = Plan(wl.x.shape, wl.w.shape, "f32")
        assert p.info()["fwd"]["kind"] == "default"
        y = host(p.forward(dev(wl.x, torch), dev(wl.w, torch)))
    assert normwise_rel(y, oracle.fwd(wl.x, wl.w)) <= 1e-5


def test_corrupt_tune_cache_is_ignored(tmp_path):
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    (tmp_path / "tune.tsv").write_bytes(b"\x00\xffgarbage\nno-tab-line\n\tempty-key\nkey-only\t\n")
    wl = inputs.random_case(3200, 30, 41, 4, 6, 3, 3)
    with _env(FBCORR_CACHE_DIR=str(tmp_path)):
        p = Plan(wl.x.shape, wl.w.shape, "f32")
        assert p.info()["fwd"]["source"] == "heuristic"
        p.autotune()                               # rewrites the cache atomically
        assert p.info()["fwd"]["source"] == "tuned"
        q = Plan(wl.x.shape, wl.w.shape, "f32")
        assert q.info()["fwd"]["source"] == "cache"
        y = host(q.forward(dev(wl.x, torch), dev(wl.w, torch)))
    assert normwise_rel(y, oracle.fwd(wl.x, wl.w)) <= 1e-5
    text = (tmp_path / "tune.tsv").read_text(errors="replace")
    assert "direct:" in text or "default" in text


F3DROP = [("f32", "f32tc:nt=32,r=1,gc=16,jt=3,ru=1"), ("f32", "f32tc:nt=64,r=2,gc=8,jt=3,ru=2"),
          ("bf16x3", "tcpack:nt=32,r=1,gc=8,jt=3,ru=2"), ("bf16", "tcpack:nt=32,r=1,gc=16,jt=3,ru=3")]


@pytest.mark.parametrize("dtype,spec", F3DROP)
def test_f32tc_dropped_copy_times_out_and_context_survives(dtype, spec):
    """FBCORR_FAULT=f3drop leaves out the first copy of the bank, for which an issuer of
    the kernel then waits in vain (here 50 ms): status, drained copies and MMAs, and a
    context on which the next plan computes."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(3300, 60, 150, 16, 32, 3, 3)
    x, w = dev(wl.x, torch), dev(wl.w, torch)
    with _env(FBCORR_FAULT="f3drop", FBCORR_WAIT_MS="50"):
        bad = Plan(wl.x.shape, wl.w.shape, dtype)
        bad.set_variant(spec)
    bad.forward(x, w)
    torch.cuda.synchronize()
    assert bad.device_status(clear=True) == 9 and bad.device_status() == 0
    good = Plan(wl.x.shape, wl.w.shape, dtype)
    good.set_variant(spec)
    y = host(good.forward(x, w))
    assert good.device_status() == 0
    assert normwise_rel(y, oracle.fwd(wl.x, wl.w)) <= (1e-2 if dtype == "bf16" else 2e-5)


@pytest.mark.parametrize("shape", [(30, 41, 16, 64, 7, 7), (21, 60, 4, 36, 2, 19)], ids=["two_planes", "tap_groups"])
def test_gradients_dropped_arrival_times_out_and_context_survives(shape):
    """The same for both gradients; dL/dw then comes from the FMA kernel behind it."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import Plan
    wl = inputs.random_case(3400, *shape, kind="int", with_g=True)
    args = [dev(t, torch) for t in (wl.x, wl.w, wl.g)]
    with _env(FBCORR_FAULT="f3drop", FBCORR_WAIT_MS="50", FBCORR_F32TC="force"):
        bad = Plan(wl.x.shape, wl.w.shape)
        for kw in ({"need_dw": False}, {"need_dx": False}):
            dw = bad.backward(*args, **kw)[1]
            torch.cuda.synchronize()
            assert bad.device_status(clear=True) == 9 and bad.device_status() == 0
    assert np.array_equal(host(dw), oracle.bwd_filt(wl.x, wl.g, wl.w.shape))
    with _env(FBCORR_F32TC="force"):
        good = Plan(wl.x.shape, wl.w.shape)
        dx, dw = good.backward(*args)
        info = good.info()
    assert info["dx"]["kind"] == "f32tc" and "f32tc" in info["dw"] and good.device_status() == 0
    assert np.array_equal(host(dx), oracle.bwd_input(wl.g, wl.w, wl.x.shape))
    assert np.array_equal(host(dw), oracle.bwd_filt(wl.x, wl.g, wl.w.shape))


def test_batch_dropped_copy_is_reported_and_does_not_refuse_the_next_call():
    """A batch kernel that gave up a wait shows in the plan's device status, which a
    single or last call can ask for after a synchronise; the next call still runs."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import BatchPlan
    items = [inputs.random_case(3500 + k, 40, 50 + 30 * k, 8, 16 * (k + 1), 3, 5, kind="int") for k in range(3)]
    shapes = [it.x.shape for it in items], [it.w.shape for it in items]
    xs, ws = [dev(it.x, torch) for it in items], [dev(it.w, torch) for it in items]
    with _env(FBCORR_FAULT="f3drop", FBCORR_WAIT_MS="50", FBCORR_F32TC="force"):
        bad = BatchPlan(*shapes)
    assert bad.info()["tensor_images"] == 3 and bad.device_status() == 0
    bad.forward(xs, ws)
    torch.cuda.synchronize()
    assert bad.device_status() == 9
    bad.forward(xs, ws)                         # not refused for what the call before it met
    torch.cuda.synchronize()
    assert bad.device_status(clear=True) == 9 and bad.device_status() == 0
    for sw in ("force", "0"):
        with _env(FBCORR_F32TC=sw):
            good = BatchPlan(*shapes)
        ys = good.forward(xs, ws)
        torch.cuda.synchronize()
        assert good.device_status() == 0
        for it, y in zip(items, ys):
            assert np.array_equal(host(y), oracle.fwd(it.x, it.w))


def test_no_device_memory_for_optional_scratch(tmp_path):
    """Where the device has no memory for scratch that a call can do without (a fake of the
    allocation that fails), tuning, batches and the host-buffer forward still run, on the
    kernels that need none, as they did before there was such scratch."""
    torch = torch_cuda()
    from paper_0911_3456_gb300.api import BatchPlan, Plan
    wl = inputs.random_case(3600, 90, 130, 8, 32, 5, 5, kind="int")
    x, w, ref = dev(wl.x, torch), dev(wl.w, torch), oracle.fwd(wl.x, wl.w)
    with _env(FBCORR_FAULT="scratchmem", FBCORR_CACHE_DIR=str(tmp_path), FBCORR_TUNE_TOPK="2", FBCORR_F32TC="force"):
        p = Plan(wl.x.shape, wl.w.shape)
        y = p.forward_host(torch.from_numpy(wl.x), torch.from_numpy(wl.w))
        torch.cuda.synchronize()
        assert p.info()["fwd"]["kind"] == "f32tc" and np.array_equal(host(y), ref)
        p.autotune()
        assert p.info()["fwd"]["source"] == "tuned" and p.info()["fwd"]["kind"] != "f32tc"
        assert np.array_equal(host(p.forward(x, w)), ref)
        b = Plan(wl.x.shape, wl.w.shape, "bf16x3")
        b.autotune()
        assert b.info()["fwd"]["spec"].startswith("tcgen05:") and np.array_equal(host(b.forward(x, w)), ref)
        batch = BatchPlan([wl.x.shape] * 2, [wl.w.shape] * 2)
        assert batch.info()["tensor_images"] == 0
        ys = batch.forward([x, x], [w, w])
        torch.cuda.synchronize()
        assert all(np.array_equal(host(t), ref) for t in ys)
