"""Performance cases of the ResNet-18 training step: the work that a program built on this
package has it do, through the package's public entry points.

A training run of the hybrid scheme is a sequence of dual-batch iterations at changing
resolutions and batch sizes, so the cases are its whole iterations (captured as a CUDA graph, as
``DualBatchIteration.capture`` does, and enqueued call by call, as the free-running workers of
``schedule.AsyncDualBatch`` are) and its parts at the sizes they have there: residual blocks forward
and backward, the stem forward (with the progressive resize) and backward, and the head.  Sizes are
those of the CIFAR-shaped (16 to 32 px) and ImageNet-shaped (128 to 288 px) workloads, in both storage
formats.  The parts are captured once as a graph and replayed, like the iteration they belong to.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2509_26092_gb300 import dbl as D
from paper_2509_26092_gb300 import resnet18 as R

EPS = 1e-5
LR, MOMENTUM, F_SMALL = 0.002, 0.9, 19.0 / 21.0  # the schedules' third learning-rate stage
DTYPE = {"bf16": torch.bfloat16, "f16": torch.float16}
WIDTHS = (64, 128, 256, 512)


# ------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the largest stage of the ImageNet-shaped hybrid run: 512 + 128 images at 224 px, one graph
        dict(name="iteration_imagenet_224", kind="iteration", variant="imagenet", res=224, native=224, large=512,
             small=128, prec="bf16"),
        # a middle stage of the CIFAR-shaped hybrid run (32 px images resized to 24 px)
        dict(name="iteration_cifar_24", kind="iteration", variant="cifar", res=24, native=32, large=512, small=128,
             prec="bf16"),
        # one small worker's step and its push, enqueued call by call (asynchronous schedule), with the loss
        # scaling of the fp16 runs: bound by launches
        dict(name="push_cifar_32_f16", kind="push", variant="cifar", res=32, native=32, large=64, prec="f16"),
        # layer1 block of the 224 px large worker: the widest maps, 64 channels
        dict(name="block_fwd_56x64_b512", kind="block_fwd", n=512, h=56, cin=64, cout=64, prec="bf16"),
        dict(name="block_bwd_56x64_b512", kind="block_bwd", n=512, h=56, cin=64, cout=64, prec="bf16"),
        # downsampling block layer3.0 of a 160 px worker, fp16 storage
        dict(name="block_fwd_down_20x256_b128_f16", kind="block_fwd", n=128, h=20, cin=128, cout=256, prec="f16"),
        # downsampling block layer2.0 of the paper's small 288 px worker's batch at 224 px: an odd batch
        dict(name="block_bwd_down_56x128_b185", kind="block_bwd", n=185, h=56, cin=64, cout=128, prec="bf16"),
        # layer4 block of a CIFAR-shaped worker (32 px: 4 x 4 maps), forward, and of a small one at 24 px
        # (3 x 3 maps), backward: the smallest layers, many channels over few pixels
        dict(name="block_fwd_4x512_b256", kind="block_fwd", n=256, h=4, cin=512, cout=512, prec="bf16"),
        dict(name="block_bwd_3x512_b64", kind="block_bwd", n=64, h=3, cin=512, cout=512, prec="bf16"),
        # the ImageNet-shaped stem at the middle resolution (8-bit 224 px images to 160 px), large worker
        dict(name="stem_fwd_160_b512", kind="stem_fwd", variant="imagenet", n=512, native=224, res=160, prec="bf16"),
        # its backward at the paper's largest resolution, the small worker's odd batch
        dict(name="stem_bwd_288_b185", kind="stem_bwd", variant="imagenet", n=185, res=288, prec="bf16"),
        # the head of the large worker, 1000 classes, with dropout
        dict(name="head_7x512_b512", kind="head", n=512, hw=49, c=512, classes=1000, drop=0.3, prec="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes over the whole range of the two workloads, odd batches included."""
    kind = rng.choice(["block_fwd", "block_fwd", "block_bwd", "block_bwd", "stem_fwd", "stem_bwd", "head", "iteration",
                       "push"])
    variant = rng.choice(["cifar", "imagenet"])
    prec = rng.choice(["bf16", "bf16", "f16"])
    res = rng.choice([16, 24, 32] if variant == "cifar" else [128, 160, 192, 224, 256, 288])
    native = 32 if variant == "cifar" else rng.choice([r for r in (224, 288) if r >= res])
    top = 1024 if variant == "cifar" else max(64, 512 * 224 * 224 // (res * res))  # the images a case may hold
    n = _log_int(rng, 16, top)
    if kind in ("block_fwd", "block_bwd"):
        layer = rng.randrange(4)
        down = layer > 0 and rng.random() < 0.4
        base = res if variant == "cifar" else res // 4
        h = base // (1 << layer) * (2 if down else 1)
        cout = WIDTHS[layer]
        return dict(kind=kind, n=n, h=h, cin=WIDTHS[layer - 1] if down else cout, cout=cout, prec=prec)
    if kind == "stem_fwd":
        return dict(kind=kind, variant=variant, n=n, native=native, res=res, prec=prec)
    if kind == "stem_bwd":
        return dict(kind=kind, variant=variant, n=n, res=res, prec=prec)
    if kind == "head":
        side = max(2, (res if variant == "cifar" else res // 4) // 8)
        return dict(kind=kind, n=n, hw=side * side, c=512, classes=100 if variant == "cifar" else 1000,
                    drop=rng.choice([0.0, 0.1, 0.2, 0.3]), prec=prec)
    if kind == "push":
        return dict(kind=kind, variant=variant, res=res, native=native, large=min(n, 128), prec=prec)
    large = max(16, min(n, 256))
    return dict(kind=kind, variant=variant, res=res, native=native, large=large, small=max(4, large // 4), prec=prec)


# ------------------------------------------------------------------------------------------ helpers
class Gen:
    """Inputs drawn on the GPU from a seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(self, shape, std=1.0, dtype=torch.float32):
        t = torch.empty(shape, device="cuda")
        return t.normal_(0.0, std, generator=self.g).to(dtype)

    def features(self, n, h, c, std, smooth, dtype):
        """Feature maps (or their gradient): noise plus a smooth pattern per image (``smooth``: [n, h, h, 1])
        that each channel takes up by its own factor, as neighbouring pixels of a network's maps share one.
        Without it every sum over pixels would be a sum of independent noise, near zero."""
        t = torch.empty((n, h, h, c), device="cuda").normal_(generator=self.g)
        return t.add_(smooth * self.normal((c,))).mul_(std).to(dtype)

    def smooth(self, n, h):
        k = (h + 3) // 4
        return F.interpolate(self.normal((n, 1, k, k)), size=(h, h)).permute(0, 2, 3, 1)

    def uniform(self, shape, lo, hi):
        return torch.empty(shape, device="cuda").uniform_(lo, hi, generator=self.g)

    def ints(self, shape, hi, dtype):
        return torch.randint(0, hi, shape, generator=self.g, device="cuda", dtype=dtype)


def _bn_params(g, c):
    """gamma and beta as a trained network has them."""
    return g.uniform((c,), 0.5, 1.5), g.normal((c,), 0.1)


def _stats(y):
    """Batch mean and 1/std of an NHWC tensor per channel, fp32."""
    f = y.reshape(-1, y.shape[-1])
    mean = f.mean(0, dtype=torch.float64)
    sq = torch.zeros_like(mean)
    for part in f.split(1 << 20):
        sq += (part.double() - mean).square().sum(0)
    return mean.float(), (1.0 / torch.sqrt(sq / f.shape[0] + EPS)).float()


def _bn_apply(y, mean, istd, gamma, beta, res=None, relu=True):
    out = (y.float() - mean) * (istd * gamma) + beta
    if res is not None:
        out += res.float()
    return (out.relu_() if relu else out).to(y.dtype)


class Graph:
    """The calls of ``body(stream)`` captured once and replayed, as the framework captures an iteration."""

    def __init__(self, body, reset=None):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            body(s.cuda_stream)
            if reset is not None:
                reset()
        torch.cuda.synchronize()
        self.g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.g, stream=s):
            body(s.cuda_stream)
        torch.cuda.synchronize()

    def replay(self):
        self.g.replay()


def _out(h, r, stride, pad):
    return (h + 2 * pad - r) // stride + 1


# ------------------------------------------------------------------------------------------ residual blocks
def _block_geometry(case):
    down = case["cin"] != case["cout"]
    stride = 2 if down else 1
    return down, stride, _out(case["h"], 3, stride, 1)


def _block_shapes(case):
    """The block's convolutions: conv1, conv2 and, for a downsampling block, the projection."""
    down, stride, ho = _block_geometry(case)
    n, h, ci, co = case["n"], case["h"], case["cin"], case["cout"]
    s1 = D.conv_shape(n, h, h, ci, co, 3, stride, 1)
    s2 = D.conv_shape(n, ho, ho, co, co, 3, 1, 1)
    return s1, s2, D.conv_shape(n, h, h, ci, co, 1, stride, 0) if down else None


def _block_weights(g, case, dt):
    ci, co = case["cin"], case["cout"]
    w = {"w1": g.normal((co, 3, 3, ci), math.sqrt(2.0 / (9 * ci)), dt),
         "w2": g.normal((co, 3, 3, co), math.sqrt(2.0 / (9 * co)), dt)}
    for k in ("1", "2"):
        w["g" + k], w["b" + k] = _bn_params(g, co)
    if ci != co:
        w["wd"] = g.normal((co, 1, 1, ci), math.sqrt(2.0 / ci), dt)
        w["gd"], w["bd"] = _bn_params(g, co)
    return w


def _block_ws(case):
    s1, s2, sd = _block_shapes(case)
    need = D.dbl_bn_workspace_bytes(D.bn_shape(case["n"] * _block_geometry(case)[2] ** 2, case["cout"]))
    for s in (s1, s2, sd):
        if s is not None:
            for ps in (D.DBL_PASS_FWD, D.DBL_PASS_DGRAD, D.DBL_PASS_WGRAD):
                need = max(need, D.dbl_conv_workspace_bytes(s, ps))
    return torch.empty(int(need) + 256, dtype=torch.uint8, device="cuda")


def _prepare_block_fwd(case, seed):
    """A block's input (the previous block's ReLU output), weights and buffers."""
    g, dt = Gen(seed), DTYPE[case["prec"]]
    down, stride, ho = _block_geometry(case)
    n, h, ci, co = case["n"], case["h"], case["cin"], case["cout"]
    st = _block_weights(g, case, dt)
    st["x"] = g.features(n, h, ci, 1.0, g.smooth(n, h), dt).relu_()
    s1, s2, sd = _block_shapes(case)

    def act():
        return torch.empty((n, ho, ho, co), dtype=dt, device="cuda")

    def vec():
        return torch.empty(co, device="cuda")

    out = {k: act() for k in ("h1", "o1", "h2", "out")}
    out.update({k: vec() for k in ("m1", "i1", "m2", "i2")})
    parts = [torch.empty(D.dbl_conv_stats_parts_bytes(s) // 4, device="cuda") for s in (s1, s2)]
    if down:
        out.update(hs=act(), sc=act(), md=vec(), id=vec())
        parts.append(torch.empty(D.dbl_conv_stats_parts_bytes(sd) // 4, device="cuda"))
    st["parts"], st["out"] = parts, out
    bn, bn_lin = D.bn_shape(n * ho * ho, co, EPS, True), D.bn_shape(n * ho * ho, co, EPS, False)

    def body(s):
        with D.precision(case["prec"]):
            k1 = D.dbl_conv_fwd_parts(s1, st["x"], st["w1"], out["h1"], parts[0], parts[0].numel() * 4, s)
            D.dbl_bn_relu_fused_parts(bn, out["h1"], parts[0], k1, st["g1"], st["b1"], None, out["o1"], out["m1"],
                                      out["i1"], s)
            k2 = D.dbl_conv_fwd_parts(s2, out["o1"], st["w2"], out["h2"], parts[1], parts[1].numel() * 4, s)
            res = st["x"]
            if down:
                kd = D.dbl_conv_fwd_parts(sd, st["x"], st["wd"], out["hs"], parts[2], parts[2].numel() * 4, s)
                D.dbl_bn_relu_fused_parts(bn_lin, out["hs"], parts[2], kd, st["gd"], st["bd"], None, out["sc"],
                                          out["md"], out["id"], s)
                res = out["sc"]
            D.dbl_bn_relu_fused_parts(bn, out["h2"], parts[1], k2, st["g2"], st["b2"], res, out["out"], out["m2"],
                                      out["i2"], s)

    st["graph"] = Graph(body)
    return st


def _prepare_block_bwd(case, seed):
    """The block's stored forward tensors, the incoming gradient, weights and buffers."""
    g, dt = Gen(seed), DTYPE[case["prec"]]
    down, stride, ho = _block_geometry(case)
    n, h, ci, co = case["n"], case["h"], case["cin"], case["cout"]
    st = _block_weights(g, case, dt)
    smooth = g.smooth(n, h)
    st["x"] = g.features(n, h, ci, 1.0, smooth, dt).relu_()
    smooth = smooth[:, ::stride, ::stride]
    st["h1"] = g.features(n, ho, co, 1.4, smooth, dt)
    st["h2"] = g.features(n, ho, co, 1.4, smooth, dt)
    st["m1"], st["i1"] = _stats(st["h1"])
    st["m2"], st["i2"] = _stats(st["h2"])
    st["o1"] = _bn_apply(st["h1"], st["m1"], st["i1"], st["g1"], st["b1"])
    res = st["x"]
    if down:
        st["hs"] = g.features(n, ho, co, 1.4, smooth, dt)
        st["md"], st["id"] = _stats(st["hs"])
        res = _bn_apply(st["hs"], st["md"], st["id"], st["gd"], st["bd"], relu=False)
    st["o"] = _bn_apply(st["h2"], st["m2"], st["i2"], st["g2"], st["b2"], res)
    # the gradient of a batch-mean loss; under fp16 it carries the loss scale.  An identity block's
    # output gradient comes in two parts (the next block's convolution and its shortcut)
    std = 1.0 if case["prec"] == "f16" else 1e-3
    st["dout"] = g.features(n, ho, co, std, smooth, dt)
    st["dout2"] = None if down else g.features(n, ho, co, std, smooth, dt)
    s1, s2, sd = _block_shapes(case)

    def act(c=co, hh=ho):
        return torch.empty((n, hh, hh, c), dtype=dt, device="cuda")

    out = {k: act() for k in ("dh2", "g", "do1", "dh1")}
    out["din"] = act(ci, h)
    out.update({k: torch.empty_like(st[k[1:]], dtype=torch.float32) for k in ("dw1", "dw2")})
    out.update({k: torch.empty(co, device="cuda") for k in ("dg1", "db1", "dg2", "db2")})
    if down:
        out.update(dhs=act(), dwd=torch.empty_like(st["wd"], dtype=torch.float32),
                   dgd=torch.empty(co, device="cuda"), dbd=torch.empty(co, device="cuda"))
    st["out"], st["ws"] = out, _block_ws(case)
    ws, wsb = st["ws"], st["ws"].numel()
    bn, bn_lin = D.bn_shape(n * ho * ho, co, EPS, True), D.bn_shape(n * ho * ho, co, EPS, False)

    def body(s):
        with D.precision(case["prec"]):
            D.dbl_bn_relu_fused_bwd(bn, st["dout"], st["dout2"], st["h2"], st["o"], st["g2"], st["m2"], st["i2"],
                                    out["dh2"], out["g"], out["dg2"], out["db2"], ws, wsb, s)
            D.dbl_conv_wgrad(s2, st["o1"], out["dh2"], out["dw2"], False, ws, wsb, s)
            D.dbl_conv_dgrad(s2, out["dh2"], st["w2"], out["do1"], None, 0, s)
            D.dbl_bn_relu_fused_bwd(bn, out["do1"], None, st["h1"], None, st["g1"], st["m1"], st["i1"], out["dh1"],
                                    None, out["dg1"], out["db1"], ws, wsb, s, beta=st["b1"])
            D.dbl_conv_wgrad(s1, st["x"], out["dh1"], out["dw1"], False, ws, wsb, s)
            if down:
                D.dbl_bn_relu_fused_bwd(bn_lin, out["g"], None, st["hs"], None, st["gd"], st["md"], st["id"],
                                        out["dhs"], None, out["dgd"], out["dbd"], ws, wsb, s)
                D.dbl_conv_wgrad(sd, st["x"], out["dhs"], out["dwd"], False, ws, wsb, s)
                D.dbl_conv_dgrad_proj(s1, out["dh1"], st["w1"], co, out["dhs"], st["wd"], out["din"], None, 0, s)
            else:
                D.dbl_conv_dgrad(s1, out["dh1"], st["w1"], out["din"], None, 0, s)

    st["graph"] = Graph(body)
    return st


# ------------------------------------------------------------------------------------------ stem
def _stem(case):
    spec = R.ResNet18Spec(case["variant"], 1000 if case["variant"] == "imagenet" else 100)
    st, lay = spec.stem, spec.stem_layout
    p = _out(case["res"], st.r, st.stride, st.pad)
    rows = lay.rows(case["res"], p)
    shape = D.conv_shape(case["n"], rows, p, 64, st.cout, lay.taps, lay.conv_stride, lay.conv_pad, s=1, stride_w=1,
                         pad_w=0)
    return spec, st, lay, p, rows, shape


def _stem_weight(g, spec, st, lay, dt):
    w = torch.zeros(lay.stored_shape(st), dtype=dt, device="cuda")
    w[:, :st.r, :st.r, :3] = g.normal((st.cout, st.r, st.r, 3), math.sqrt(2.0 / (st.r * st.r * 3)), dt)
    return w


def _prepare_stem_fwd(case, seed):
    """8-bit images at the native resolution, the stem's weights and buffers."""
    g, dt = Gen(seed), DTYPE[case["prec"]]
    spec, cs, lay, p, rows, shape = _stem(case)
    n, nat = case["n"], case["native"]
    st = {"img": g.ints((n, nat, nat, 3), 256, torch.uint8), "w": _stem_weight(g, spec, cs, lay, dt)}
    st["g"], st["b"] = _bn_params(g, 64)
    ws = torch.empty(int(D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_FWD)) + 256, dtype=torch.uint8, device="cuda")
    out = {"x0": torch.empty((n, rows, p, 64), dtype=dt, device="cuda"),
           "y": torch.empty((n, p, p, 64), dtype=dt, device="cuda")}
    out.update({k: torch.empty(64, device="cuda") for k in ("sum", "sumsq", "mean", "istd")})
    q = _out(p, 3, 2, 1)
    if case["variant"] == "imagenet":
        out["a"] = torch.empty((n, q, q, 64), dtype=dt, device="cuda")
        out["arg"] = torch.empty((n, q, q, 64), dtype=torch.uint8, device="cuda")
    else:
        out["a"] = torch.empty((n, p, p, 64), dtype=dt, device="cuda")
    st["out"], st["ws"] = out, ws
    bn = D.bn_shape(n * p * p, 64, EPS, True)
    res = case["res"]

    def body(s):
        with D.precision(case["prec"]):
            D.dbl_progressive_resize_stem_u8(st["img"], n, nat, nat, 3, R.PIXEL_SCALE, R.PIXEL_BIAS, out["x0"], res,
                                             res, cs.r, cs.stride, cs.pad, lay.rg, lay.pad_h, rows, s)
            D.dbl_conv_fwd(shape, out["x0"], st["w"], out["y"], out["sum"], out["sumsq"], ws, ws.numel(), s)
            if case["variant"] == "imagenet":
                D.dbl_bn_relu_maxpool_fwd(bn, n, p, p, out["y"], out["sum"], out["sumsq"], st["g"], st["b"],
                                          out["mean"], out["istd"], out["a"], out["arg"], s)
            else:
                D.dbl_bn_relu_fused(bn, out["y"], out["sum"], out["sumsq"], st["g"], st["b"], None, out["a"],
                                    out["mean"], out["istd"], s)

    st["graph"] = Graph(body)
    return st


def _prepare_stem_bwd(case, seed):
    """The stem's stored input and output, the incoming gradient (in two parts, from the first
    block's convolution and its shortcut) and buffers."""
    g, dt = Gen(seed), DTYPE[case["prec"]]
    spec, cs, lay, p, rows, shape = _stem(case)
    n = case["n"]
    imagenet = case["variant"] == "imagenet"
    st = {"x0": g.normal((n, rows, p, 64), 1.0, dt), "y": g.normal((n, p, p, 64), 1.2, dt)}
    st["g"], st["b"] = _bn_params(g, 64)
    st["m"], st["i"] = _stats(st["y"])
    q = _out(p, 3, 2, 1) if imagenet else p
    std = 1.0 if case["prec"] == "f16" else 1e-3
    st["dout"], st["dout2"] = g.normal((n, q, q, 64), std, dt), g.normal((n, q, q, 64), std, dt)
    if imagenet:
        args = []
        at = 2 * torch.arange(q, device="cuda") - 1  # first row / column of each window
        for y in st["y"].split(32):  # the argmax of the pooled BatchNorm output, as its forward pass leaves it
            a = _bn_apply(y, st["m"], st["i"], st["g"], st["b"]).float().permute(0, 3, 1, 2)
            idx = F.max_pool2d(a, 3, 2, 1, return_indices=True)[1]
            k = (idx // p - at[:, None]) * 3 + (idx % p - at[None, :])
            args.append(k.permute(0, 2, 3, 1).to(torch.uint8))
        st["arg"] = torch.cat(args).contiguous()
    need = max(D.dbl_conv_workspace_bytes(shape, D.DBL_PASS_WGRAD), D.dbl_bn_workspace_bytes(D.bn_shape(n * p * p, 64)))
    ws = torch.empty(int(need) + 256, dtype=torch.uint8, device="cuda")
    out = {"dy": torch.empty((n, p, p, 64), dtype=dt, device="cuda"),
           "dw": torch.empty(lay.stored_shape(cs), device="cuda"),
           "dg": torch.empty(64, device="cuda"), "db": torch.empty(64, device="cuda")}
    if imagenet:
        out["da"] = torch.empty((n, p, p, 64), dtype=dt, device="cuda")
    st["out"], st["ws"] = out, ws
    bn = D.bn_shape(n * p * p, 64, EPS, True)

    def body(s):
        with D.precision(case["prec"]):
            da, da2 = st["dout"], st["dout2"]
            if imagenet:
                D.dbl_maxpool_bwd(n, p, p, 64, st["dout"], st["dout2"], st["arg"], out["da"], s)
                da, da2 = out["da"], None
            D.dbl_bn_relu_fused_bwd(bn, da, da2, st["y"], None, st["g"], st["m"], st["i"], out["dy"], None, out["dg"],
                                    out["db"], ws, ws.numel(), s, beta=st["b"])
            D.dbl_conv_wgrad(shape, st["x0"], out["dy"], out["dw"], False, ws, ws.numel(), s)

    st["graph"] = Graph(body)
    return st


# ------------------------------------------------------------------------------------------ head
HEAD_SEED, HEAD_STEP = 77, 5


def _prepare_head(case, seed):
    """The last block's output (after ReLU), the FC parameters, labels and buffers."""
    g, dt = Gen(seed), DTYPE[case["prec"]]
    n, hw, c, j = case["n"], case["hw"], case["c"], case["classes"]
    st = {"x": g.normal((n, hw, c), 1.0).relu_().to(dt), "fc_w": g.normal((j, c), math.sqrt(2.0 / c)),
          "fc_b": g.normal((j,), 0.1), "lab": g.ints((n,), j, torch.int32),
          "step": torch.full((1,), HEAD_STEP, dtype=torch.int64, device="cuda"),
          "scale": torch.full((1,), 2.0 ** 15, device="cuda") if case["prec"] == "f16" else None}
    out = {"loss": torch.empty(1, device="cuda"), "dfc_w": torch.empty((j, c), device="cuda"),
           "dfc_b": torch.empty(j, device="cuda"), "dx": torch.empty((n, hw, c), dtype=dt, device="cuda")}
    ws = torch.empty(int(D.dbl_head_workspace_bytes(n, c, j)) + 256, dtype=torch.uint8, device="cuda")
    st["out"], st["ws"] = out, ws

    def body(s):
        with D.precision(case["prec"]):
            opts = D.head_opts(case["drop"], HEAD_SEED, st["step"] if case["drop"] > 0 else None, st["scale"])
            D.dbl_head_fwd_bwd_ex(n, hw, c, j, st["x"], st["fc_w"], st["fc_b"], st["lab"], opts, out["loss"],
                                  out["dfc_w"], out["dfc_b"], out["dx"], ws, ws.numel(), s)

    st["graph"] = Graph(body, reset=lambda: st["step"].fill_(HEAD_STEP))
    return st


# ------------------------------------------------------------------------------------------ whole steps
def _server(case, g):
    spec = R.ResNet18Spec(case["variant"], 1000 if case["variant"] == "imagenet" else 100)
    params, vel = {}, {}
    for name, shape, fan_in in spec.table():
        if fan_in is not None:
            params[name] = g.normal(shape, math.sqrt(2.0 / fan_in))
        else:
            params[name] = torch.ones(shape, device="cuda") if name.endswith(".g") else torch.zeros(shape, device="cuda")
        vel[name] = g.normal(shape, 0.01)  # momentum, as in the middle of a run
    return spec, R.ServerState(spec, params, vel, precision=case["prec"])


def _worker(case, spec, server, n, g, tag):
    wk = R.Worker(spec, n, case["res"], dropout=0.2, dropout_seed=tag, precision=case["prec"])
    img = g.ints((n, case["native"], case["native"], 3), 256, torch.uint8)
    return wk, img, g.ints((n,), spec.classes, torch.int32)


def _prepare_iteration(case, seed):
    """The server's model, both workers and the captured dual-batch iteration on their images."""
    g = Gen(seed)
    spec, server = _server(case, g)
    large, img_l, lab_l = _worker(case, spec, server, case["large"], g, 1)
    small, img_s, lab_s = _worker(case, spec, server, case["small"], g, 2)
    it = R.DualBatchIteration(server, large, small, case["native"], lr=LR, momentum=MOMENTUM, f_small=F_SMALL)
    it.set_inputs(img_l, lab_l, img_s, lab_s)
    it.capture()
    return {"server": server, "it": it, "large": large, "small": small}


def _prepare_push(case, seed):
    """The server's model and one worker with its images: the step is enqueued call by call."""
    g = Gen(seed)
    spec, server = _server(case, g)
    wk, img, lab = _worker(case, spec, server, case["large"], g, 1)
    wk.labels.copy_(lab)
    return {"server": server, "worker": wk, "img": img, "native": case["native"]}


PREPARE = {"block_fwd": _prepare_block_fwd, "block_bwd": _prepare_block_bwd, "stem_fwd": _prepare_stem_fwd,
           "stem_bwd": _prepare_stem_bwd, "head": _prepare_head, "iteration": _prepare_iteration,
           "push": _prepare_push}


def prepare(case, seed):
    st = PREPARE[case["kind"]](case, seed)
    st["kind"] = case["kind"]
    return st


def run(st):
    if st["kind"] == "iteration":
        st["it"].run()
        return {"w": st["server"].w, "u": st["server"].u, "loss_large": st["large"].loss, "loss_small": st["small"].loss}
    if st["kind"] == "push":
        server, wk = st["server"], st["worker"]
        stream = torch.cuda.current_stream()
        wk.enqueue_step(server, st["img"], st["native"], stream)
        server.apply_pushes(wk.grad, None, wk.scale_used, None, LR, MOMENTUM, 1.0, F_SMALL, 0, stream.cuda_stream)
        return {"w": server.w, "u": server.u, "loss": wk.loss}
    st["graph"].replay()
    return st["out"]


# ------------------------------------------------------------------------------------------ work
def work(case):
    """Bytes: every input read once, every output written once.  FLOPs: 2*M*N*K of each GEMM."""
    kind = case["kind"]
    if kind in ("block_fwd", "block_bwd"):
        down, stride, ho = _block_geometry(case)
        n, h, ci, co = case["n"], case["h"], case["cin"], case["cout"]
        x, o = n * h * h * ci, n * ho * ho * co
        wts = 9 * ci * co + 9 * co * co + (ci * co if down else 0)
        f = 2 * n * ho * ho * wts
        if kind == "block_fwd":
            return {"bytes": 2 * (x + wts + (6 if down else 4) * o), "flops": f}
        reads = 2 * (x + (6 if down else 6) * o + wts)  # x, o1, h1, h2, o, dout and dout2 or hs, weights
        writes = 2 * ((5 if down else 4) * o + x) + 4 * wts
        return {"bytes": reads + writes, "flops": 2 * f}
    if kind in ("stem_fwd", "stem_bwd"):
        spec, cs, lay, p, rows, _ = _stem(case)
        n = case["n"]
        x0, y = n * rows * p * 64, n * p * p * 64
        imagenet = case["variant"] == "imagenet"
        a = n * _out(p, 3, 2, 1) ** 2 * 64 if imagenet else y
        f = 2 * n * p * p * 64 * cs.r * cs.r * 3
        if kind == "stem_fwd":
            return {"bytes": n * case["native"] ** 2 * 3 + 2 * (x0 + y + a) + (a if imagenet else 0), "flops": f}
        return {"bytes": 2 * (x0 + y + 2 * a + y) + ((a + 2 * y) if imagenet else 0), "flops": f}
    if kind == "head":
        n, hw, c, j = case["n"], case["hw"], case["c"], case["classes"]
        return {"bytes": 2 * 2 * n * hw * c + 2 * 4 * j * c, "flops": 6 * n * c * j}
    spec = R.ResNet18Spec(case["variant"], 1000 if case["variant"] == "imagenet" else 100)
    images = case["large"] + case.get("small", 0)
    f, h = 0, _out(case["res"], spec.stem.r, spec.stem.stride, spec.stem.pad)
    f += 2 * 2 * h * h * 64 * spec.stem.r ** 2 * 3
    h = _out(h, 3, 2, 1) if case["variant"] == "imagenet" else h
    for b in spec.blocks:
        ho = _out(h, 3, b.stride, 1)
        f += 3 * 2 * ho * ho * (9 * b.cin * b.cout + 9 * b.cout ** 2 + (b.cin * b.cout if b.proj else 0))
        h = ho
    return {"bytes": images * case["native"] ** 2 * 3 + 4 * 4 * spec.n_params(), "flops": images * f}


# ------------------------------------------------------------------------------------------ tolerance
def tolerance(case):
    """About four times what the passes show with their sums in another order (torch's fp32
    convolutions and sums with the same 16-bit storage points for the parts; an epsilon that moves
    1/std by 1e-6 for whole steps).  A sum in another order moves a stored 16-bit value by one rounding
    step here and there, at most 2^-8 (bf16) or 2^-11 (f16) of the value, and by a few at the end of a
    chain of layers.  A whole step's gradient amplifies that about a hundred times, and its updated
    weights carry it into the next step."""
    f16 = case["prec"] == "f16"
    kind = case["kind"]
    if kind in ("iteration", "push"):
        return {"rel": 0.012, "max": 0.7}
    if kind == "head":
        return {"rel": 1e-4 if f16 else 4e-4, "max": 0.004 if f16 else 0.02}
    if kind in ("stem_fwd", "stem_bwd"):
        return {"rel": 2e-4 if f16 else 1e-3, "max": 0.02 if f16 else 0.1, "differ": 1e-3}
    return {"rel": 5e-4 if f16 else 3e-3, "max": 0.02 if f16 else 0.1}


# ------------------------------------------------------------------------------------------ 64 bits
def _conv64(x, w, stride, pad):
    """NHWC x, KRSC w (fp64) -> NHWC."""
    return F.conv2d(x.permute(0, 3, 1, 2), w.permute(0, 3, 1, 2), stride=stride, padding=pad).permute(0, 2, 3, 1)


def _dgrad64(dy, w, hw, stride, pad):
    shape = (dy.shape[0], w.shape[3], hw, hw)
    return torch.nn.grad.conv2d_input(shape, w.permute(0, 3, 1, 2), dy.permute(0, 3, 1, 2), stride=stride,
                                      padding=pad).permute(0, 2, 3, 1)


def _wgrad64(x, dy, wshape, stride, pad):
    k, r, s, c = wshape
    return torch.nn.grad.conv2d_weight(x.permute(0, 3, 1, 2), (k, c, r, s), dy.permute(0, 3, 1, 2), stride=stride,
                                       padding=pad).permute(0, 2, 3, 1)


def _bn64(y, gamma, beta):
    f = y.reshape(-1, y.shape[-1])
    mean, var = f.mean(0), f.var(0, unbiased=False)
    istd = 1.0 / torch.sqrt(var + EPS)
    return (y - mean) * (istd * gamma.double()) + beta.double(), mean, istd


def _bn_bwd64(g, y, mean, istd, gamma):
    c = y.shape[-1]
    xhat = (y - mean.double()) * istd.double()
    db, dg = g.reshape(-1, c).sum(0), (g * xhat).reshape(-1, c).sum(0)
    n = g.numel() // c
    return gamma.double() * istd.double() * (g - db / n - xhat * (dg / n)), dg, db


def _exact_block_fwd(case, st):
    down, stride, _ = _block_geometry(case)
    x = st["x"].double()
    e = {"h1": _conv64(x, st["w1"].double(), stride, 1)}
    a, e["m1"], e["i1"] = _bn64(e["h1"], st["g1"], st["b1"])
    e["o1"] = a.relu_()
    e["h2"] = _conv64(e["o1"], st["w2"].double(), 1, 1)
    a, e["m2"], e["i2"] = _bn64(e["h2"], st["g2"], st["b2"])
    if down:
        e["hs"] = _conv64(x, st["wd"].double(), stride, 0)
        e["sc"], e["md"], e["id"] = _bn64(e["hs"], st["gd"], st["bd"])
        x = e["sc"]
    e["out"] = (a + x).relu_()
    return e


def _exact_block_bwd(case, st):
    down, stride, _ = _block_geometry(case)
    h = case["h"]
    g = st["dout"].double()
    if st["dout2"] is not None:
        g = g + st["dout2"].double()
    g = g * (st["o"] > 0)
    e = {"g": g}
    e["dh2"], e["dg2"], e["db2"] = _bn_bwd64(g, st["h2"].double(), st["m2"], st["i2"], st["g2"])
    w1, w2 = st["w1"].double(), st["w2"].double()
    e["dw2"] = _wgrad64(st["o1"].double(), e["dh2"], w2.shape, 1, 1)
    e["do1"] = _dgrad64(e["dh2"], w2, e["dh2"].shape[1], 1, 1)
    h1 = st["h1"].double()
    sc = st["g1"].double() * st["i1"].double()
    mask = h1 * sc + (st["b1"].double() - st["m1"].double() * sc) > 0
    e["dh1"], e["dg1"], e["db1"] = _bn_bwd64(e["do1"] * mask, h1, st["m1"], st["i1"], st["g1"])
    x = st["x"].double()
    e["dw1"] = _wgrad64(x, e["dh1"], w1.shape, stride, 1)
    e["din"] = _dgrad64(e["dh1"], w1, h, stride, 1)
    if down:
        e["dhs"], e["dgd"], e["dbd"] = _bn_bwd64(g, st["hs"].double(), st["md"], st["id"], st["gd"])
        e["dwd"] = _wgrad64(x, e["dhs"], st["wd"].shape, stride, 0)
        e["din"] = e["din"] + _dgrad64(e["dhs"], st["wd"].double(), h, stride, 0)
    return e


def _resize64(img, res):
    """Half-pixel bilinear downsampling with edge clamp of standardized NHWC pixels, fp64."""
    sc = torch.tensor(R.PIXEL_SCALE, dtype=torch.float64, device="cuda")
    x = img.double() * sc + torch.tensor(R.PIXEL_BIAS, dtype=torch.float64, device="cuda")
    nat = img.shape[1]
    num = (2 * torch.arange(res, device="cuda") + 1) * nat - res
    i0 = num // (2 * res)
    i1 = (i0 + 1).clamp(max=nat - 1)
    lam = (num - i0 * 2 * res).double() / (2 * res)
    x = x[:, i0] * (1 - lam)[:, None, None] + x[:, i1] * lam[:, None, None]
    return x[:, :, i0] * (1 - lam)[:, None] + x[:, :, i1] * lam[:, None]


def _exact_stem_fwd(case, st):
    spec, cs, lay, p, rows, _ = _stem(case)
    n, res = case["n"], case["res"]
    e = {k: None for k in st["out"]}
    cu = 8 // lay.rg
    x0 = torch.zeros((n, rows, p, lay.rg, 8, cu), dtype=torch.float64, device="cuda")
    y = torch.empty((n, p, p, 64), dtype=torch.float64, device="cuda")
    w = st["w"][:, :cs.r, :cs.r, :3].double()
    q_at = cs.stride * torch.arange(p, device="cuda")
    m_at = lay.rg * torch.arange(rows, device="cuda")
    for k in range(0, n, 64):
        img = _resize64(st["img"][k:k + 64], res)
        y[k:k + 64] = _conv64(img, w, cs.stride, cs.pad)
        pad = F.pad(img, (0, 0, cs.pad, 8, lay.pad_h, 8))
        for r in range(lay.rg):
            for t in range(cs.r):
                x0[k:k + 64, :, :, r, t, :3] = pad[:, m_at + r][:, :, q_at + t]
    e["x0"], e["y"] = x0.reshape(n, rows, p, 64), y
    f = y.reshape(-1, 64)
    e["sum"], e["sumsq"] = f.sum(0), f.square().sum(0)
    a, e["mean"], e["istd"] = _bn64(y, st["g"], st["b"])
    a.relu_()
    if case["variant"] == "imagenet":
        a = torch.cat([F.max_pool2d(t.permute(0, 3, 1, 2), 3, 2, 1).permute(0, 2, 3, 1) for t in a.split(64)])
    e["a"] = a
    return e


def _exact_stem_bwd(case, st):
    spec, cs, lay, p, rows, _ = _stem(case)
    n = case["n"]
    e = {}
    da = st["dout"].double() + st["dout2"].double()
    if case["variant"] == "imagenet":
        q = da.shape[1]
        full = torch.zeros((n, p + 2, p + 2, 64), dtype=torch.float64, device="cuda")  # one pixel of padding
        for k in range(9):
            full[:, k // 3:k // 3 + 2 * q:2, k % 3:k % 3 + 2 * q:2][:, :q, :q] += da * (st["arg"] == k)
        da = full[:, 1:p + 1, 1:p + 1].contiguous()
        e["da"] = da
    y = st["y"].double()
    sc = st["g"].double() * st["i"].double()
    g = da * (y * sc + (st["b"].double() - st["m"].double() * sc) > 0)
    e["dy"], e["dg"], e["db"] = _bn_bwd64(g, y, st["m"], st["i"], st["g"])
    dw = torch.zeros((64, lay.taps, 64), dtype=torch.float64, device="cuda")
    x = F.pad(st["x0"], (0, 0, 0, 0, lay.conv_pad, lay.conv_pad))
    dy = e["dy"]
    for k in range(0, n, 16):  # taps x 1 stride-1 convolution of the unrolled input
        d = dy[k:k + 16].reshape(-1, 64)
        for t in range(lay.taps):
            dw[:, t] += d.t() @ x[k:k + 16, t:t + p].double().reshape(-1, 64)
    e["dw"] = dw.reshape(lay.stored_shape(cs))
    return e


def _keep(n, c, drop):
    """The dropout mask: word c % 4 of Philox4x64-10 block n*c/4 + c/4, kept when its upper half is large."""
    raw = np.random.Philox(counter=(HEAD_STEP << 64) - 1, key=HEAD_SEED).random_raw(n * c)
    return torch.from_numpy((raw >> np.uint64(32)) >= np.uint64(math.floor(float(np.float32(drop)) * 2 ** 32))
                            ).reshape(n, c).cuda()


def _exact_head(case, st):
    n, hw, c = case["n"], case["hw"], case["c"]
    feat = st["x"].double().mean(1)
    mult = torch.ones_like(feat)
    if case["drop"] > 0:
        mult = _keep(n, c, case["drop"]).double() / (1.0 - float(np.float32(case["drop"])))
    feat = feat * mult
    w, lab = st["fc_w"].double(), st["lab"].long()
    logits = feat @ w.t() + st["fc_b"].double()
    loss = F.cross_entropy(logits, lab).reshape(1)
    dl = torch.softmax(logits, 1)
    dl[torch.arange(n, device="cuda"), lab] -= 1.0
    dl *= (float(st["scale"]) if st["scale"] is not None else 1.0) / n
    dx = ((dl @ w) * mult / hw)[:, None, :].expand(n, hw, c)
    return {"loss": loss, "dfc_w": dl.t() @ feat, "dfc_b": dl.sum(0), "dx": dx}


EXACT = {"block_fwd": _exact_block_fwd, "block_bwd": _exact_block_bwd, "stem_fwd": _exact_stem_fwd,
         "stem_bwd": _exact_stem_bwd, "head": _exact_head}


def exact(case, seed):
    f = EXACT.get(case["kind"])
    if f is None:  # a whole step stores 16-bit values layer by layer; its parts are held to 64 bits
        return None
    return f(case, prepare(case, seed))
