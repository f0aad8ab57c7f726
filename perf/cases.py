"""Performance cases of the filter-bank correlation library.

Each case is one call (or one training step) of the public Python entry points on
device tensors, with plans as a program gets them by default (no tuning run).  The
shapes are those of the repository's workloads (``inputs.py``, ``bench.py``): the
paper's table of filter-bank shapes, the precision workload, the differentiation
workload, the batch of uneven images, the three-layer cascade and the
nearest-neighbour search, beside odd sizes of the same ranges.
"""
import math

import torch

from paper_0911_3456_gb300 import BatchPlan, NNPlan, Plan, fbcorr
from paper_0911_3456_gb300.cascade import Cascade, Layer

LEAK = "y > 0.f ? y : lo * y"   # the cascade's static non-linearity
LEAK_SLOPE = 0.1


def listed():
    return [
        # the smallest image of the uneven batches alone, with a small bank: what one call costs
        _fwd("patch_f32", 64, 64, 4, 16, 3, 3),
        # the repository's first configuration: one small image of a model's first layer
        _fwd("small_f32", 128, 128, 8, 16, 9, 9, bank="unit"),
        # row 1 of the paper's table with the clamp of its models' non-linearity
        _fwd("paper_row1_clamp_f32", 256, 256, 8, 64, 9, 9, bank="unit", clamp=True),
        # row 4 of the paper's table: a large image, few channels and few filters
        _fwd("paper_row4_f32", 2048, 2048, 4, 4, 8, 8, bank="unit"),
        # the precision workload in the three arithmetics a user chooses from
        _fwd("dense_f32", 512, 512, 32, 256, 5, 5),
        _fwd("dense_bf16x3", 512, 512, 32, 256, 5, 5, dtype="bf16x3"),
        # odd sizes of an image that comes from elsewhere, in plain BF16
        _fwd("ragged_bf16", 301, 419, 24, 96, 7, 5, dtype="bf16"),
        # the differentiation workload as an autograd training step: y, dL/dx and dL/dw
        {"name": "train_f32", "kind": "train", "H": 256, "W": 256, "D": 16, "N": 64, "fh": 7, "fw": 7},
        # the gradients of a clamped layer of odd sizes (the masked kernels)
        {"name": "backward_clamp_f32", "kind": "backward", "H": 187, "W": 233, "D": 12, "N": 40, "fh": 5, "fw": 3},
        # images of uneven sizes, each with its own bank, in one call
        {"name": "batch_f32", "kind": "batch", "count": 24, "shapes_seed": 4},
        # the three-layer model structure: bank, fused non-linearity, next bank
        {"name": "cascade_bf16x3", "kind": "cascade", "H": 256, "W": 256, "D": 8, "dtype": "bf16x3"},
        # the exact nearest-neighbour search of the paper's second study
        {"name": "nn_search", "kind": "nn", "targets": 4096, "neighbors": 262144, "side": 8, "dtype": "bf16x3"},
    ]


def _fwd(name, H, W, D, N, fh, fw, dtype="f32", clamp=False, bank="scaled"):
    c = {"kind": "forward", "H": H, "W": W, "D": D, "N": N, "fh": fh, "fw": fw, "dtype": dtype, "clamp": clamp,
         "bank": bank}
    return dict({"name": name}, **c) if name else c


# ---------------------------------------------------------------- drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _layer(rng, max_flops, max_depth=64):
    """Image, depth, bank and filter sizes of one layer within a FLOP limit."""
    while True:
        H, W = _log(rng, 32, 2048), _log(rng, 32, 2048)
        D = rng.choice([4, 8, 16, 32, _log(rng, 1, max_depth)])
        N = rng.choice([16, 32, 64, 128, _log(rng, 4, 256)])
        fh = rng.randint(3, 13)
        fw = fh if rng.random() < 0.6 else rng.randint(3, 13)
        if fh > H or fw > W or H * W * max(D, N) > 1 << 27:
            continue
        if 2 * (H - fh + 1) * (W - fw + 1) * N * fh * fw * D <= max_flops:
            return {"H": H, "W": W, "D": D, "N": N, "fh": fh, "fw": fw}


def draw(rng):
    kind = rng.choices(["forward", "train", "backward", "batch", "cascade", "nn"], [11, 3, 2, 1, 1, 2])[0]
    if kind == "forward":
        dtype = rng.choices(["f32", "bf16x3", "bf16"], [6, 3, 2])[0]
        s = _layer(rng, 6e10, 64 if dtype == "f32" else 32)
        return _fwd(None, s["H"], s["W"], s["D"], s["N"], s["fh"], s["fw"], dtype, rng.random() < 0.3,
                    rng.choice(["scaled", "unit"]))
    if kind in ("train", "backward"):
        return dict({"kind": kind}, **_layer(rng, 1.2e10, 32))
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(4, 24), "shapes_seed": rng.randint(5, 10 ** 6)}
    if kind == "cascade":
        return {"kind": "cascade", "H": _log(rng, 96, 384), "W": _log(rng, 96, 384), "D": rng.choice([4, 8, 12]),
                "dtype": rng.choice(["f32", "bf16x3"])}
    return {"kind": "nn", "targets": _log(rng, 256, 4096), "neighbors": _log(rng, 4096, 262144),
            "side": rng.choice([5, 6, 8]), "dtype": "bf16x3"}


# ---------------------------------------------------------------- inputs
def _uniform(shape, gen, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=gen, device="cuda") * (hi - lo) + lo


def _bank(shape, gen, how):
    """"unit": zero mean and unit L2 norm per filter; "scaled": variance 1 / (fh fw D)."""
    w = torch.randn(shape, generator=gen, device="cuda")
    if how == "unit":
        w = w - w.mean(dim=(1, 2, 3), keepdim=True)
        return w / w.square().sum(dim=(1, 2, 3), keepdim=True).sqrt()
    return w / math.sqrt(shape[1] * shape[2] * shape[3])


BATCH_HW = tuple(range(64, 513, 32))


def _batch_shapes(case):
    gen = torch.Generator().manual_seed(case["shapes_seed"])

    def pick(values):
        return values[int(torch.randint(len(values), (1,), generator=gen))]

    out = []
    for _ in range(case["count"]):
        H, W, D = pick(BATCH_HW), pick(BATCH_HW), pick((4, 8, 16, 32))
        N, f = pick((16, 32, 64, 128)), pick((3, 5, 7, 9, 11))
        out.append(((H, W, D), (N, f, f, D)))
    return out


CASCADE_BANKS = ((64, 9, 9), (32, 5, 5), (16, 3, 3))


def _patches(count, side, gen, images, size=512):
    """Rows of side x side patches cut at random places of images with the 1/f
    amplitude spectrum of natural scenes, scaled to [0, 1]."""
    fy = torch.fft.fftfreq(size, device="cuda")[:, None]
    fx = torch.fft.rfftfreq(size, device="cuda")[None, :]
    f = (fx * fx + fy * fy).sqrt()
    f[0, 0] = 1.0
    phase = torch.rand((images,) + tuple(f.shape), generator=gen, device="cuda") * (2 * math.pi)
    img = torch.fft.irfft2(torch.polar((1.0 / f).expand_as(phase), phase), s=(size, size))
    lo, hi = img.amin(dim=(1, 2), keepdim=True), img.amax(dim=(1, 2), keepdim=True)
    flat = ((img - lo) / (hi - lo)).reshape(-1)
    span = size - side + 1
    k = torch.randint(images, (count, 1), generator=gen, device="cuda")
    r = torch.randint(span, (count, 1), generator=gen, device="cuda")
    c = torch.randint(span, (count, 1), generator=gen, device="cuda")
    off = (torch.arange(side, device="cuda")[:, None] * size + torch.arange(side, device="cuda")).reshape(1, -1)
    return flat[k * size * size + r * size + c + off].contiguous()


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind == "nn":
        neighbors = _patches(case["neighbors"], case["side"], gen, 7)
        return {"targets": _patches(case["targets"], case["side"], gen, 1), "neighbors": neighbors}
    if kind == "batch":
        shapes = _batch_shapes(case)
        return {"xs": [_uniform(a, gen) for a, _ in shapes],
                "ws": [torch.randn(b, generator=gen, device="cuda") for _, b in shapes]}
    H, W, D = case["H"], case["W"], case["D"]
    if kind == "cascade":
        x, banks, depth = _uniform((H, W, D), gen), [], D
        for n, fh, fw in CASCADE_BANKS:
            banks.append(_bank((n, fh, fw, depth), gen, "unit"))
            depth = n
        return {"x": x, "banks": banks}
    N, fh, fw = case["N"], case["fh"], case["fw"]
    x = _uniform((H, W, D), gen, -1.0 if case.get("bank") == "scaled" else 0.0, 1.0)
    d = {"x": x, "w": _bank((N, fh, fw, D), gen, case.get("bank", "scaled"))}
    if kind in ("train", "backward"):
        d["g"] = torch.randn((H - fh + 1, W - fw + 1, N), generator=gen, device="cuda")
    if kind == "backward":   # the layer's forward output, as its program has it
        d["y"] = _corr64(d["x"], d["w"]).clamp(*CLAMP).float()
    return d


CLAMP = (0.0, 1.0)


def prepare(case, seed):
    s = dict(_inputs(case, seed), kind=case["kind"])
    kind = case["kind"]
    if kind == "forward":
        s["plan"] = Plan(s["x"].shape, s["w"].shape, case["dtype"], CLAMP if case["clamp"] else None)
    elif kind == "backward":
        s["plan"] = Plan(s["x"].shape, s["w"].shape, "f32", CLAMP)
    elif kind == "train":
        s["x"].requires_grad_()
        s["w"].requires_grad_()
    elif kind == "batch":
        s["plan"] = BatchPlan([x.shape for x in s["xs"]], [w.shape for w in s["ws"]])
    elif kind == "cascade":
        layers = [Layer(n, fh, fw, LEAK, (LEAK_SLOPE, 0.0)) for n, fh, fw in CASCADE_BANKS]
        s["plan"] = Cascade(s["x"].shape, layers, case["dtype"])
    else:
        s["plan"] = NNPlan(case["targets"], case["neighbors"], case["side"] ** 2, case["dtype"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "forward":
        return s["plan"].forward(s["x"], s["w"])
    if kind == "backward":
        return s["plan"].backward(s["x"], s["w"], s["g"], s["y"])
    if kind == "train":
        y = fbcorr(s["x"], s["w"], "f32")
        dx, dw = torch.autograd.grad(y, (s["x"], s["w"]), s["g"])
        return y.detach(), dx, dw
    if kind == "batch":
        return s["plan"].forward(s["xs"], s["ws"])
    if kind == "cascade":
        return s["plan"].forward(s["x"], s["banks"])
    return s["plan"].search(s["targets"], s["neighbors"])


# ---------------------------------------------------------------- work and 64-bit values
def _layer_work(H, W, D, N, fh, fw):
    Ho, Wo = H - fh + 1, W - fw + 1
    return H * W * D, N * fh * fw * D, Ho * Wo * N, 2.0 * Ho * Wo * N * fh * fw * D


def work(case):
    kind = case["kind"]
    if kind == "nn":
        t, n, dim = case["targets"], case["neighbors"], case["side"] ** 2
        return {"bytes": 4 * (t + n) * dim + 12 * t, "flops": 3.0 * t * n * dim}
    if kind == "batch":
        parts = [_layer_work(*a, b[0], b[1], b[2]) for a, b in _batch_shapes(case)]
        return {"bytes": 4 * sum(x + w + y for x, w, y, _ in parts), "flops": sum(p[3] for p in parts)}
    if kind == "cascade":
        H, W, D = case["H"], case["W"], case["D"]
        nbytes, flops = 4 * H * W * D, 0.0
        for n, fh, fw in CASCADE_BANKS:
            _, w, y, f = _layer_work(H, W, D, n, fh, fw)
            H, W, D = H - fh + 1, W - fw + 1, n
            nbytes += 4 * w
            flops += f
        return {"bytes": nbytes + 4 * y, "flops": flops}
    x, w, y, f = _layer_work(*(case[k] for k in ("H", "W", "D", "N", "fh", "fw")))
    if kind == "forward":
        return {"bytes": 4 * (x + w + y), "flops": f}
    if kind == "train":     # reads x, w, g; writes y, dx, dw
        return {"bytes": 8 * (x + w + y), "flops": 3 * f}
    return {"bytes": 4 * (2 * x + 2 * w + 2 * y), "flops": 2 * f}   # backward: reads x, w, g, y; writes dx, dw


def _corr64(x, w):
    x, w = x.detach().double(), w.detach().double()
    N, fh, fw, D = w.shape
    Ho, Wo = x.shape[0] - fh + 1, x.shape[1] - fw + 1
    y = torch.zeros((Ho * Wo, N), dtype=torch.float64, device=x.device)
    for i in range(fh):
        for j in range(fw):
            y.addmm_(x[i:i + Ho, j:j + Wo].reshape(-1, D), w[:, i, j].t())
    return y.reshape(Ho, Wo, N)


def _grads64(x, w, g):
    x, w, g = x.detach().double(), w.detach().double(), g.double()
    N, fh, fw, D = w.shape
    Ho, Wo = g.shape[:2]
    dx, dw, gf = torch.zeros_like(x), torch.zeros_like(w), g.reshape(-1, N)
    for i in range(fh):
        for j in range(fw):
            dx[i:i + Ho, j:j + Wo] += (gf @ w[:, i, j]).reshape(Ho, Wo, D)
            dw[:, i, j] = gf.t() @ x[i:i + Ho, j:j + Wo].reshape(-1, D)
    return dx, dw


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "forward":
        y = _corr64(d["x"], d["w"])
        return y.clamp(*CLAMP) if case["clamp"] else y
    if kind == "backward":
        inside = (d["y"] > CLAMP[0]) & (d["y"] < CLAMP[1])
        return _grads64(d["x"], d["w"], d["g"] * inside)
    if kind == "train":
        return (_corr64(d["x"], d["w"]),) + _grads64(d["x"], d["w"], d["g"])
    if kind == "batch":
        return [_corr64(x, w) for x, w in zip(d["xs"], d["ws"])]
    if kind == "cascade":
        h = d["x"].double()
        for w in d["banks"]:
            h = _corr64(h, w)
            h = torch.where(h > 0, h, float(torch.tensor(LEAK_SLOPE)) * h)
        return h
    t, n = d["targets"].double(), d["neighbors"].double()
    best = [((t[a:a + 512].square().sum(1)[:, None] + n.square().sum(1)[None, :] - 2 * t[a:a + 512] @ n.t()).argmin(1))
            for a in range(0, len(t), 512)]
    return None, (t - n[torch.cat(best)]).square().sum(1)
