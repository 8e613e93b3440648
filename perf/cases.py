"""The work that is timed: PSB layers and whole networks through the public entry points.

A case is one of three kinds.

  fc    one fully connected layer: ``Context.sample_weights`` (fresh draws) and ``Context.gemm``
  conv  one convolution, dense or depthwise: ``Context.sample_weights`` and ``Context.conv2d``
  net   a whole network: ``Network.sample`` and ``Network.forward`` (and, in the two-pass scheme of
        Sec. 4.5, ``Context.attention_entropy`` and ``Context.attention_maps`` between two passes)

``resample`` says whether a pass draws its filters anew, as every inference of the paper does
(Sec. 4.1), or uses the filters sampled before (a service that keeps one set of draws).  Sampling
twice under one seed gives the same filters, so the outputs of a case depend on the seed alone.
Everything random is made on the GPU from the seed; the quantisation steps follow in closed form
from the layer shapes, so that no calibration pass is needed.
"""
import math

import numpy as np
import torch

import paper_1904_02205_b200 as psb
from paper_1904_02205_b200.network import Network
from workloads import mobilenetv2_layers, network_macs, resnet50_layers, tiny_mobilenet_layers, tiny_resnet_layers

_FC = dict(kind="fc", log2k=2, act_max=15, signed_in=False, norm=0, exp_bits=4, underflow=0, prob_bits=0, out="q",
           resample=True)
_CONV = dict(kind="conv", groups="dense", ksize=3, stride=1, pad=1, log2k=3, per_location=False, layout="nhwc",
             act_max=15, signed_in=False, residual=False, out="q", norm=0, exp_bits=4, underflow=0, prob_bits=0,
             resample=True)
_NET = dict(kind="net", log2k=3, mode="uniform")

_ARCH = {"resnet50": (resnet50_layers, 224, 15, 15, 0.0),          # 4-bit activations
         "mobilenetv2": (mobilenetv2_layers, 224, 255, 127, 0.5),  # 8-bit activations, half of the weights pruned
         "tiny_resnet": (tiny_resnet_layers, 40, 15, 15, 0.0),
         "tiny_mobilenet": (tiny_mobilenet_layers, 32, 255, 127, 0.5)}
_LAST = {"resnet50": "s4b2_out", "tiny_resnet": "s2b0_out", "mobilenetv2": "head", "tiny_mobilenet": "head"}
_MAP_LEVELS = 0b11111                       # k = 1, 2, 4, 8, 16
_MAP_QUANTILES = (0.30, 0.55, 0.80, 0.925)  # share of the locations below each threshold: mean k = 4


def listed():
    return [
        # a small classifier head, fresh draws for every batch: the smallest call, all latency
        dict(_FC, name="fc_256x128_b16", batch=16, d_in=256, d_out=128, act_max=15),
        # the 1000-class head of a network on one request, filters kept, real-valued logits wanted
        dict(_FC, name="fc_2048x1000_b1_logits", batch=1, d_in=2048, d_out=1000, log2k=3, out="f32", resample=False),
        # a wide hidden layer at serving batch, 8-bit probabilities, one window per output channel, unbiased floor
        dict(_FC, name="fc_4096x4096_b256", batch=256, d_in=4096, d_out=4096, log2k=4, act_max=127, norm=1,
             underflow=1, prob_bits=8),
        # the layer that the benchmark quotes, planar tensors in and out
        dict(_CONV, name="conv3x3_64_56_b32_planar", n=32, c=64, o=64, h=56, w=56, layout="nchw"),
        # the expanding 1x1 layer with the shortcut added, the class with the most bytes per operation
        dict(_CONV, name="conv1x1_64_256_56_b64_shortcut", n=64, c=64, o=256, h=56, w=56, ksize=1, pad=0, residual=True,
             resample=False),
        # channel counts as they come out of channel pruning, an image that is no square, 8-bit activations
        dict(_CONV, name="conv3x3_100_150_57x43_b7_8bit", n=7, c=100, o=150, h=57, w=43, act_max=255, log2k=4),
        # a depthwise layer of an inverted residual, 8-bit activations
        dict(_CONV, name="depthwise3x3_144_56_b64", n=64, c=144, o=144, h=56, w=56, groups="depthwise", act_max=255,
             log2k=4),
        # one image through the large network: latency of a whole forward pass
        dict(_NET, name="resnet50_b1", arch="resnet50", batch=1),
        # throughput, uniform draw counts
        dict(_NET, name="resnet50_b64", arch="resnet50", batch=64),
        # throughput, draw counts per location from a given saliency map: the largest call
        dict(_NET, name="resnet50_b128_map", arch="resnet50", batch=128, mode="map"),
        # two passes, the second one refined where the first was undecided (Sec. 4.5)
        dict(_NET, name="resnet50_b32_attention", arch="resnet50", batch=32, mode="attention"),
        # the depthwise-separable network at 8 bits
        dict(_NET, name="mobilenetv2_b64", arch="mobilenetv2", batch=64, log2k=4),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Half of the time a multiple of 16, half of the time whatever comes."""
    c = _log_uniform(rng, lo, hi)
    return max(16, (c + 8) // 16 * 16) if rng.random() < 0.5 else c


def _sampling_options(rng):
    return dict(norm=rng.choice([0, 1]), exp_bits=rng.choice([4, 4, 3]), underflow=rng.choice([0, 1]),
                prob_bits=rng.choice([0, 0, 4, 8]), resample=rng.random() < 0.6)


def draw(rng):
    kind = rng.choice(["fc", "conv", "conv", "net"])
    if kind == "fc":
        return dict(_FC, batch=_log_uniform(rng, 1, 512), d_in=_channels(rng, 64, 4096), d_out=_channels(rng, 10, 4096),
                    log2k=rng.randint(0, 4), act_max=rng.choice([15, 127, 255]), out=rng.choice(["q", "q", "f32"]),
                    **_sampling_options(rng))
    if kind == "conv":
        groups = rng.choice(["dense", "dense", "dense", "depthwise"])
        ksize = rng.choice([3, 3, 5]) if groups == "depthwise" else rng.choice([1, 1, 3, 3, 3, 5, 7])
        h = _log_uniform(rng, 7, 112)
        w = h if rng.random() < 0.5 else max(7, int(h * rng.uniform(0.5, 1.5)))
        c = 3 if ksize == 7 else _channels(rng, 16, 512)
        o = c if groups == "depthwise" else _channels(rng, 16, 768)
        stride = 2 if ksize == 7 else rng.choice([1, 1, 2])
        act_max = rng.choice([15, 15, 255, 127])
        case = dict(_CONV, groups=groups, ksize=ksize, stride=stride, pad=ksize // 2, c=c, o=o, h=h, w=w,
                    log2k=rng.randint(0, 4), per_location=rng.random() < 0.2, layout=rng.choice(["nhwc", "nhwc", "nchw"]),
                    act_max=act_max, signed_in=act_max == 127 and rng.random() < 0.5, residual=rng.random() < 0.3,
                    out=rng.choice(["q", "q", "q", "q+f32"]), **_sampling_options(rng))
        # at most 5e10 multiply-accumulates and 2e8 input bytes
        per_image = _conv_macs(dict(case, n=1))
        most = min(5e10 / per_image, 2e8 / (c * h * w), 128)
        return dict(case, n=_log_uniform(rng, 1, max(1.0, most)))
    arch = rng.choice(["resnet50", "mobilenetv2", "tiny_resnet", "tiny_mobilenet"])
    mode = rng.choice(["uniform", "uniform", "map", "attention"]) if arch == "resnet50" else "uniform"
    return dict(_NET, arch=arch, batch=_log_uniform(rng, 1, 48 if mode == "attention" else 128), mode=mode,
                log2k=3 if mode == "attention" else rng.randint(0, 4))


# --------------------------------------------------------------------------- inputs

_contexts = {}


def _context():
    """A program keeps one context per device."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = psb.Context(dev)
    return _contexts[dev]


class _State:
    """What a program holds between calls; gives the library's device memory back when it is dropped."""

    def __init__(self, case, **kw):
        self.case = case
        self.__dict__.update(kw)

    def __del__(self):
        for name in ("weights", "second", "net"):
            held = getattr(self, name, None)
            if held is not None:
                held.free()


def _normal(gen, shape, std):
    return torch.empty(shape, device="cuda").normal_(0.0, std, generator=gen)


def _codes(gen, shape, act_max, signed):
    """Activations after a ReLU: half zeros, the rest uniform in [1, act_max]; signed: uniform in [-act_max, act_max]."""
    if signed:
        return torch.randint(-act_max, act_max + 1, shape, generator=gen, device="cuda", dtype=torch.int8)
    x = torch.randint(1, act_max + 1, shape, generator=gen, device="cuda", dtype=torch.uint8)
    return x * torch.randint(0, 2, shape, generator=gen, device="cuda", dtype=torch.uint8)


def _mean_square(act_max, signed):
    return act_max * act_max / (3.0 if signed else 6.0)


def _field_maps(gen, n, shapes, ref):
    """Draw-count maps (log2 k = 0..4) of every (h, w) in `shapes` from a smooth random saliency field per image:
    three Gaussian blobs, thresholds at fixed quantiles of the field on the `ref` grid."""
    def uni(lo, hi):
        return torch.empty((n, 3, 1, 1), device="cuda", dtype=torch.float64).uniform_(lo, hi, generator=gen)

    cx, cy, width, height = uni(0.0, 1.0), uni(0.0, 1.0), uni(0.08, 0.25), uni(0.5, 1.0)

    def field(h, w):
        v = ((torch.arange(h, device="cuda", dtype=torch.float64) + 0.5) / h).view(1, 1, h, 1)
        u = ((torch.arange(w, device="cuda", dtype=torch.float64) + 0.5) / w).view(1, 1, 1, w)
        return (height * torch.exp(-((u - cx) ** 2 + (v - cy) ** 2) / (2 * width ** 2))).sum(1)

    flat = field(*ref).flatten(1).sort(dim=1).values
    thr = [flat[:, min(flat.shape[1] - 1, int(q * flat.shape[1]))].view(n, 1, 1) for q in _MAP_QUANTILES]
    maps = {}
    for hw in shapes:
        f = field(*hw)
        maps[hw] = sum((f > t).to(torch.uint8) for t in thr)
    return maps


def _relu_moments(mu, var):
    """(mean, mean square) of max(y, 0) for y ~ N(mu, var)."""
    s = math.sqrt(var)
    cdf = 0.5 * (1.0 + math.erf(mu / s / math.sqrt(2.0)))
    pdf = math.exp(-0.5 * (mu / s) ** 2) / math.sqrt(2.0 * math.pi)
    return mu * cdf + s * pdf, (mu * mu + var) * cdf + mu * s * pdf


def _network_inputs(layers, in_hw, batch, gen, qmax_u, qmax_s, prune):
    """Seeded parameters of a layer list in the form ``Network`` takes: He-normal filters (the smallest magnitudes
    of a layer pruned), folded batch-norm factors U(0.5, 1.5), output steps from the second moments that such
    filters give layer by layer."""
    image = torch.randint(0, 256, (batch, in_hw, in_hw, 3), generator=gen, device="cuda", dtype=torch.uint8)
    steps, dtypes = {"image": 1.0 / 128}, {"image": psb.PSB_DT_U8}
    moments = {"image": (127.5 / 128, 255.0 * 511 / 6 / 128 ** 2)}       # (mean, mean square)
    params, lid = {}, 0
    for l in layers:
        mean, m2 = moments[l["src"]]
        if l["op"] == "maxpool":
            moments[l["dst"]], steps[l["dst"]], dtypes[l["dst"]] = (2.6 * mean, 3.0 * m2), steps[l["src"]], dtypes[l["src"]]
            continue
        if l["op"] == "avgpool":
            out_step = 3.0 * mean / qmax_u
            params[l["name"]] = dict(pool_mul=np.float32(steps[l["src"]] / l["hin"] ** 2 / out_step), qmin=0, qmax=qmax_u)
            moments[l["dst"]], steps[l["dst"]], dtypes[l["dst"]] = (mean, 1.2 * mean * mean), out_step, psb.PSB_DT_U8
            continue
        cin_g = l["cin"] // l["groups"]
        d = cin_g * l["k"] ** 2
        w = _normal(gen, (l["cout"], cin_g, l["k"], l["k"]), math.sqrt(2.0 / d))
        if prune:
            w = torch.where(w.abs() <= 0.6745 * math.sqrt(2.0 / d), torch.zeros_like(w), w)      # the median magnitude
        bn = torch.empty(l["cout"], device="cuda").uniform_(0.5, 1.5, generator=gen)
        mu, var = 0.0, 2.0 * m2 * (13.0 / 12.0) * (0.93 if prune else 1.0) * (0.79 if l["groups"] > 1 else 1.0)
        res_scale = 0.0
        if l["residual"] is not None:
            res_scale = steps[l["residual"]]
            rm, r2 = moments[l["residual"]]
            mu, var = rm, var + r2 - rm * rm
        if l["relu"]:
            out_moments, out_step = _relu_moments(mu, var), (mu + 3.1 * math.sqrt(var)) / qmax_u
        else:
            out_moments, out_step = (mu, mu * mu + var), (abs(mu) + 3.1 * math.sqrt(var)) / qmax_s
        signed = l["signed_out"]
        params[l["name"]] = dict(
            w=w.cpu().numpy(), scale=(bn * steps[l["src"]]).cpu().numpy(), bias=_normal(gen, (l["cout"],), 0.1 * out_step).cpu().numpy(),
            inv_step=np.float32(1.0 / out_step), qmin=-qmax_s if signed else 0, qmax=qmax_s if signed else qmax_u,
            res_scale=np.float32(res_scale), layer_id=lid, out_dtype=psb.PSB_DT_S8 if signed else psb.PSB_DT_U8,
            in_dtype=dtypes[l["src"]], res_dtype=None if l["residual"] is None else dtypes[l["residual"]])
        moments[l["dst"]], steps[l["dst"]] = out_moments, out_step
        dtypes[l["dst"]] = params[l["name"]]["out_dtype"]
        lid += 1
    return dict(image=image, params=params, steps=steps, dtypes=dtypes)


def _out_hw(c):
    return (c["h"] + 2 * c["pad"] - c["ksize"]) // c["stride"] + 1, (c["w"] + 2 * c["pad"] - c["ksize"]) // c["stride"] + 1


def _conv_macs(c):
    oh, ow = _out_hw(c)
    return c["n"] * oh * ow * c["o"] * (1 if c["groups"] == "depthwise" else c["c"]) * c["ksize"] ** 2


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    ctx = _context()
    if case["kind"] == "net":
        return _prepare_net(case, seed, gen, ctx)
    opts = {k: case[k] for k in ("norm", "exp_bits", "underflow", "prob_bits")}
    if case["kind"] == "fc":
        o, cin_g, ksize, groups, per_location = case["d_out"], case["d_in"], 1, 1, False
    else:
        groups = case["c"] if case["groups"] == "depthwise" else 1
        o, cin_g, ksize, per_location = case["o"], case["c"] // groups, case["ksize"], case["per_location"]
    d = cin_g * ksize * ksize
    w = _normal(gen, (o, cin_g, ksize, ksize), math.sqrt(2.0 / d))
    scale = torch.empty(o, device="cuda").uniform_(0.5, 1.5, generator=gen)
    std = math.sqrt(2.0 * _mean_square(case["act_max"], case["signed_in"]) * 13.0 / 12.0)
    kw = dict(w=w, scale=scale, bias=_normal(gen, (o,), 0.1 * std), opts=opts, groups=groups, seed=seed)
    kw["mask"] = _MAP_LEVELS if per_location else 1 << case["log2k"]
    if case["kind"] == "fc":
        qmax = 255
        kw["x"] = _codes(gen, (case["batch"], case["d_in"]), case["act_max"], case["signed_in"])
    else:
        qmax = case["act_max"]
        n, c, h, ww = case["n"], case["c"], case["h"], case["w"]
        oh, ow = _out_hw(case)
        planar = case["layout"] == "nchw"
        kw["layout"] = psb.PSB_LAYOUT_NCHW if planar else psb.PSB_LAYOUT_NHWC
        kw["x"] = _codes(gen, (n, c, h, ww) if planar else (n, h, ww, c), case["act_max"], case["signed_in"])
        kw["map"] = _field_maps(gen, n, [(oh, ow)], (oh, ow))[(oh, ow)] if per_location else None
        kw["residual"] = None
        if case["residual"]:
            kw["residual"] = _codes(gen, (n, o, oh, ow) if planar else (n, oh, ow, o), 15, False)
        kw["residual_scale"] = 0.2 * std
    kw["qmax"], kw["inv_step"] = qmax, qmax / (3.1 * std)
    kw["want"] = tuple(case["out"].split("+"))
    kw["weights"] = ctx.sample_weights(w, groups=groups, seed=seed, layer_id=0, level_mask=kw["mask"], **opts)
    return _State(case, **kw)


def _prepare_net(case, seed, gen, ctx):
    make, in_hw, qmax_u, qmax_s, prune = _ARCH[case["arch"]]
    layers, batch, log2k = make(), case["batch"], case["log2k"]
    inputs = _network_inputs(layers, in_hw, batch, gen, qmax_u, qmax_s, prune)
    sizes = sorted({l["hout"] for l in layers if l["op"] == "conv"} - {1}, reverse=True)
    kw = dict(image=inputs["image"], seed=seed, last=_LAST[case["arch"]], second=None)
    if case["mode"] == "map":
        maps = _field_maps(gen, batch, [(r, r) for r in sizes], (sizes[1], sizes[1]))
        kw["net"] = Network(ctx, layers, inputs, batch, _MAP_LEVELS, kmaps={r[0]: m.cpu().numpy() for r, m in maps.items()},
                            fc_log2k=4)
    elif case["mode"] == "attention":
        # k = 8 everywhere, then 16 where the first pass was undecided; one set of draws serves both passes
        kw["net"] = Network(ctx, layers, inputs, batch, 0b11000, uniform_log2k=3)
        flat = {r: np.full((batch, r, r), 3, dtype=np.uint8) for r in sizes}
        kw["second"] = Network(ctx, layers, inputs, batch, 0b11000, kmaps=flat, uniform_log2k=3, fc_log2k=4,
                               weights_from=kw["net"])
        kw["sizes"], kw["last_step"] = sizes, float(inputs["steps"][kw["last"]])
    else:
        kw["net"] = Network(ctx, layers, inputs, batch, 1 << log2k, uniform_log2k=log2k)
    kw["net"].sample(seed)
    return _State(case, **kw)


# --------------------------------------------------------------------------- one pass

def run(state):
    case, ctx = state.case, _context()
    if case["kind"] == "net":
        return _run_net(state, ctx)
    if case["resample"]:
        ctx.sample_weights(state.w, groups=state.groups, seed=state.seed, layer_id=0, level_mask=state.mask,
                           into=state.weights, **state.opts)
    if case["kind"] == "fc":
        ctx.set_sample_map(None, case["log2k"])
        return ctx.gemm(state.weights, state.x, state.scale, state.bias, True, state.inv_step, 0, state.qmax,
                        in_max=case["act_max"], want=state.want)
    ctx.set_sample_map(state.map, case["log2k"])
    return ctx.conv2d(state.weights, state.x, state.layout, case["stride"], case["pad"], state.scale, state.bias, True,
                      state.inv_step, 0, state.qmax, residual=state.residual, residual_scale=state.residual_scale,
                      in_max=case["act_max"], want=state.want)


def _run_net(state, ctx):
    net = state.net
    net.sample(state.seed)
    logits = net.forward(state.image)
    out = dict(logits=logits, codes=net.acts["logits"], features=net.acts[state.last])
    if state.second is not None:
        out = {k + "_first": v for k, v in out.items()}
        entropy = ctx.attention_entropy(net.acts[state.last], state.last_step)
        ctx.attention_maps(entropy, 3, 4, state.sizes, out=state.second.kmaps)
        logits = state.second.forward(state.image)
        out.update(entropy=entropy, logits=logits, codes=state.second.acts["logits"], features=state.second.acts[state.last])
    return out


# --------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Bytes: activations in, filters (fp32 where they are drawn anew, else 4 bytes of sampled integer), per-channel
    constants, shortcut and maps in, outputs out.  Flops: two per logical multiply-accumulate, whatever number of
    digit planes carries it; the random numbers are not counted."""
    if case["kind"] == "fc":
        b, i, o = case["batch"], case["d_in"], case["d_out"]
        return {"bytes": b * i + 4 * i * o + 8 * o + b * o * (4 if case["out"] == "f32" else 1), "flops": 2 * b * i * o}
    if case["kind"] == "conv":
        oh, ow = _out_hw(case)
        outs = case["n"] * oh * ow * case["o"]
        filters = case["o"] * (1 if case["groups"] == "depthwise" else case["c"]) * case["ksize"] ** 2
        per_out = len(case["out"].split("+")) * 4 - 3 + (1 if case["residual"] else 0)
        return {"bytes": case["n"] * case["c"] * case["h"] * case["w"] + 4 * filters + 8 * case["o"] + outs * per_out
                + (case["n"] * oh * ow if case["per_location"] else 0), "flops": 2 * _conv_macs(case)}
    make, in_hw = _ARCH[case["arch"]][:2]
    layers, batch = make(), case["batch"]
    convs = [l for l in layers if l["op"] == "conv"]
    params = sum(l["cout"] * (l["cin"] // l["groups"]) * l["k"] ** 2 + 2 * l["cout"] for l in convs)
    last = next(l for l in layers if l["dst"] == _LAST[case["arch"]])
    outs = batch * (convs[-1]["cout"] * 5 + last["hout"] ** 2 * last["cout"])
    maps = batch * sum(r * r for r in {l["hout"] for l in convs} - {1}) if case["mode"] == "map" else 0
    passes = 2 if case["mode"] == "attention" else 1
    return {"bytes": batch * in_hw * in_hw * 3 + 4 * params + passes * outs + maps,
            "flops": 2 * passes * batch * network_macs(layers)}


def tolerance(case):
    """Filters, accumulators and codes are whole numbers and the same in every correct implementation; the real-valued
    outputs take correctly rounded operations only, one fma more or less apart.  The entropies of the two-pass scheme
    are fp32 sums of up to 2048 terms (measured: the location nearest to its image's mean is 5 % away, so that no
    summation order moves one across)."""
    if case["kind"] == "net":
        return {"rel": 1e-5 if case["mode"] == "attention" else 1e-6}
    return "exact" if case["out"] == "q" else {"rel": 1e-6}
