"""The workloads whose speed counts: what a program that serves column-wise N:M pruned networks has this library do.

Backbones at the batch sizes of interactive and of throughput serving, single layers under a tuned plan and under the
library's default, the general kernels' odd shapes, host buffers, and the two ways a compressed layer comes into being
(pruning dense weights, loading a checkpoint).  Layer shapes are those of ``paper_2507_17301_b200.inputs`` and generic ones.
"""
import math

import torch

from paper_2507_17301_b200 import inputs, nm


def _net(name, depth, batch, n, m, tile, image=224):
    return {"name": name, "kind": "net", "depth": depth, "batch": batch, "image": image, "n": n, "m": m, "tile": tile}


def _conv(name, batch, h, w, c_in, c_out, k, stride, pad, dil, n, m, tile, relu=True, residual=False, tuned=True, kind="conv"):
    return {"name": name, "kind": kind, "batch": batch, "h": h, "w": w, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride,
            "pad": pad, "dil": dil, "n": n, "m": m, "tile": tile, "relu": relu, "residual": residual, "tuned": tuned}


def listed():
    return [
        # the smallest call: one small layer, library default, output allocated by the call (config_tiny)
        _conv("tiny3x3_default", 1, 14, 14, 16, 32, 3, 1, 1, 1, 2, 4, 8, tuned=False),
        # one image at a time through a whole backbone: interactive serving, bound by launches and latency
        _net("resnet50_b1", 50, 1, 2, 4, 64),
        # a few images through a basic-block network (all 3x3), the paper's best case, at 75 % sparsity
        _net("resnet18_1of4_b8", 18, 8, 1, 4, 32),
        # throughput serving: the benchmark's network, batch, pattern and tile width
        _net("resnet50_b64", 50, 64, 2, 4, 64),
        # the largest: deep network, large batch, groups of eight
        _net("resnet101_2of8_b128", 101, 128, 2, 8, 64),
        # pointwise layers whose channel counts are mostly no multiples of 32 or 64
        {"name": "mobilenet_pointwise_b32", "kind": "pointwise", "batch": 32, "image": 224, "n": 2, "m": 4, "tile": 16},
        # one 3x3 layer tuned on its own (config_resnet3x3)
        _conv("c3x3_256_2of8_b32", 32, 14, 14, 256, 256, 3, 1, 1, 1, 2, 8, 32),
        # the last layer of a residual block, shortcut fused, at 87.5 % sparsity (config_bottleneck1x1)
        _conv("c1x1_256_1024_1of8_res_b64", 64, 14, 14, 256, 1024, 1, 1, 0, 1, 1, 8, 64, residual=True),
        # a user's own layer without tuning: ragged image, strided and dilated, 3:4
        _conv("ragged3x3_3of4_default", 5, 61, 75, 96, 80, 3, 2, 2, 2, 3, 4, 16, tuned=False),
        # activations in pinned host memory: upload, layer, download
        _conv("host3x3_b8", 8, 28, 28, 128, 128, 3, 1, 1, 1, 2, 4, 64, kind="host"),
        # compressing a layer: dense weights -> handle -> values and indices
        {"name": "prune_3x3_512", "kind": "prune", "c_out": 512, "k": 3, "c_in": 512, "n": 2, "m": 4, "tile": 64},
        # loading a compressed layer from a checkpoint
        {"name": "import_1x1_1024_2048", "kind": "import", "c_out": 2048, "k": 1, "c_in": 1024, "n": 2, "m": 4, "tile": 64},
    ]


_PATTERNS = ((1, 4), (2, 4), (3, 4), (1, 8), (2, 8), (4, 8))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("net", "net", "net", "conv", "conv", "conv", "pointwise", "host", "prune", "import"))
    n, m = rng.choice(_PATTERNS)
    tile = rng.choice((8, 16, 32, 64, 128))
    if kind == "net":
        depth, image = rng.choice((18, 34, 50, 101)), rng.randint(96, 288)
        return _without_name(_net("", depth, _log(rng, 1, min(128, 128 * 224 * 224 // (image * image))), n, m, tile, image))
    if kind == "pointwise":
        return {"kind": kind, "batch": _log(rng, 1, 128), "image": rng.randint(96, 224), "n": n, "m": m, "tile": 16}
    if kind in ("prune", "import"):
        return {"kind": kind, "c_out": 4 * _log(rng, 4, 512), "k": rng.choice((1, 1, 3, 3, 5)), "c_in": 4 * _log(rng, 4, 256),
                "n": n, "m": m, "tile": tile}
    k, dil = rng.choice((1, 1, 3, 3, 3, 5, 7)), rng.choice((1, 1, 1, 2))
    c_in, c_out = _log(rng, 3, 1024), 4 * _log(rng, 4, 256)
    if rng.random() < 0.7:    # most layers have whole blocks of channels
        c_in, c_out = -(-c_in // 32) * 32, -(-c_out // 32) * 32
    h, w = _log(rng, 7, 112), _log(rng, 7, 112)
    batch = _log(rng, 1, 64)
    while batch > 1 and 2e-9 * batch * h * w * c_in * c_out * k * k > 400:   # no dearer than a large layer of the listed networks
        batch //= 2
    stride, relu = rng.choice((1, 1, 1, 2)), rng.random() < 0.5
    residual = kind == "conv" and rng.random() < 0.3
    return _without_name(_conv("", batch, h, w, c_in, c_out, k, stride, dil * (k // 2), dil, n, m, tile, relu, residual,
                               rng.random() < 0.6, kind))


def _without_name(case):
    return {key: v for key, v in case.items() if key != "name"}


def _layer(case):
    return inputs.ConvShape("layer", case["batch"], case["h"], case["w"], case["c_in"], case["c_out"], case["k"], case["k"],
                            case["stride"], case["pad"], case["dil"], case["n"], case["m"], case["tile"], case["relu"])


def _layers(case):
    if case["kind"] == "net":
        return inputs.resnet_conv_stack(case["depth"], case["batch"], case["n"], case["m"], case["tile"], case["image"])
    return inputs.mobilenet_v2_pointwise(case["batch"], case["n"], case["m"], case["tile"], case["image"])


def _normal(gen, *shape, std=1.0):
    return torch.randn(shape, generator=gen, device="cuda") * std


def _weights(gen, s):
    return _normal(gen, s.c_out, s.kh, s.kw, s.c_in, std=(2.0 / s.k) ** 0.5)


class _Conv:
    """One layer of a program: pruned weights, bias, output buffer and the plan found for it."""

    def __init__(self, s, gen, plans=None, x=None):
        self.s = s
        self.hnd = nm.nm_prune(_weights(gen, s), s.n_keep, s.m_group, s.tile_t)
        self.bias = _normal(gen, s.c_out)
        self.plan = None
        if plans is not None:    # layers of the same shape share a plan
            key = (s.h, s.w, s.c_in, s.c_out, s.kh, s.stride, s.n_keep)
            if key not in plans:
                x = _normal(gen, s.batch, s.h, s.w, s.c_in) if x is None else x
                plans[key] = nm.nm_autotune(self.hnd, x, s.stride, s.pad, s.dil, self.bias, s.relu, None, s.kh, s.kw)[0]
            else:
                need = nm.nm_plan_scratch_bytes(self.hnd, (s.batch, s.h, s.w, s.c_in), s.stride, s.pad, s.dil, plans[key])
                nm.nm_weights_reserve(self.hnd, need)
            self.plan = plans[key]

    def __call__(self, x, relu, residual=None, y=None):
        s = self.s
        return nm.nm_conv2d(self.hnd, x, s.kh, s.kw, s.stride, s.pad, s.dil, self.bias, relu, y, self.plan, residual)


def _blocks(layers):
    """The residual blocks of a network: (stage, [indices of the main path], index of the projection or None)."""
    blocks = {}
    for i, s in enumerate(layers[1:], 1):
        blocks.setdefault(s.name.split("_")[0], {})[s.name.split("_")[1]] = i
    return [(pre.split("b")[0], [b[k] for k in sorted(b) if k != "ds"], b.get("ds")) for pre, b in blocks.items()]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("net", "pointwise"):
        layers, plans = _layers(case), {}
        state["convs"] = convs = [_Conv(s, gen, plans) for s in layers]
        if kind == "pointwise":
            state["x"] = [_normal(gen, s.batch, s.h, s.w, s.c_in) for s in layers]
            state["y"] = [torch.empty((s.batch, s.ho, s.wo, s.c_out), device="cuda") for s in layers]
            return state
        stem = layers[0]
        state["x"] = _normal(gen, stem.batch, stem.h, stem.w, stem.c_in)
        state["blocks"] = _blocks(layers)
        new = lambda s: torch.empty((s.batch, s.ho, s.wo, s.c_out), device="cuda")  # noqa: E731
        first = layers[1]
        state["stem_y"] = new(stem)
        state["pool_y"] = torch.empty((first.batch, first.h, first.w, first.c_in), device="cuda")
        # buffers of a stage: the shortcut, the inner maps of a block, two maps that the blocks' outputs alternate between
        state["buf"] = buf = {}
        for stage, path, ds in state["blocks"]:
            for j, i in enumerate(path):
                s = convs[i].s
                last = j + 1 == len(path)
                for key in ([(stage, "out", 0), (stage, "out", 1)] if last else [(stage, j, s.h)]):
                    if key not in buf:
                        buf[key] = new(s)
            if ds is not None:
                buf[(stage, "ds")] = new(convs[ds].s)
        return state
    if kind in ("prune", "import"):
        w = _normal(gen, case["c_out"], case["k"], case["k"], case["c_in"], std=(2.0 / (case["k"] ** 2 * case["c_in"])) ** 0.5)
        state["case"] = case
        state["w"] = w if kind == "prune" else None
        if kind == "import":
            state["values"], state["indices"] = nm.nm_weights_export(nm.nm_prune(w, case["n"], case["m"], case["tile"]))
        return state
    s = _layer(case)
    state["x"] = x = _normal(gen, s.batch, s.h, s.w, s.c_in)
    state["conv"] = _Conv(s, gen, {} if case["tuned"] else None, x)
    state["residual"] = _normal(gen, s.batch, s.ho, s.wo, s.c_out) if case["residual"] else None
    if kind == "host":
        state["x_host"] = x.cpu().pin_memory()
        state["bias_host"] = state["conv"].bias.cpu().pin_memory()
        state["y"] = torch.empty((s.batch, s.ho, s.wo, s.c_out), device="cuda")
        state["y_host"] = torch.empty(state["y"].shape, pin_memory=True)
    return state


def run(state):
    kind = state["kind"]
    if kind == "net":
        return _run_net(state)
    if kind == "pointwise":
        return [conv(x, conv.s.relu, y=y) for conv, x, y in zip(state["convs"], state["x"], state["y"])]
    if kind == "prune":
        c = state["case"]
        return nm.nm_weights_export(nm.nm_prune(state["w"], c["n"], c["m"], c["tile"]))
    if kind == "import":
        c = state["case"]
        return nm.nm_weights_export(nm.nm_weights_import(state["values"], state["indices"], c["k"], c["k"], c["c_in"], c["n"],
                                                         c["m"], c["tile"]))
    conv = state["conv"]
    if kind == "host":
        s = conv.s
        nm.nm_conv2d_host(conv.hnd, state["x_host"], state["x"], s.stride, s.pad, s.dil, state["bias_host"], conv.bias, s.relu,
                          state["y_host"], state["y"], conv.plan)
        return state["y_host"]
    return conv(state["x"], conv.s.relu, state["residual"])


def _run_net(state):
    """The convolution backbone in dataflow order; returns the feature map of every stage."""
    convs, buf = state["convs"], state["buf"]
    cur = convs[0](state["x"], True, y=state["stem_y"])
    cur = nm.nm_maxpool2d(cur, 3, 2, 1, y=state["pool_y"])
    maps, turn = {}, 0
    for stage, path, ds in state["blocks"]:
        shortcut = cur if ds is None else convs[ds](cur, False, y=buf[(stage, "ds")])
        for j, i in enumerate(path[:-1]):
            cur = convs[i](cur, True, y=buf[(stage, j, convs[i].s.h)])
        turn ^= 1
        cur = maps[stage] = convs[path[-1]](cur, True, shortcut, buf[(stage, "out", turn)])
    return list(maps.values())


def _conv_work(s, residual=False):
    read = s.pixels * s.c_in if s.kh == 1 and s.stride > 1 else s.batch * s.h * s.w * s.c_in
    tiles = -(-s.c_out // s.tile_t)
    out = s.pixels * s.c_out
    return 4 * (read + out * (2 if residual else 1) + s.c_out * s.kk + s.c_out) + 2 * tiles * s.kk, 2.0 * out * s.kk


def work(case):
    kind = case["kind"]
    if kind in ("prune", "import"):
        k = case["k"] ** 2 * case["c_in"]
        kk = k // case["m"] * case["n"] + min(k % case["m"], case["n"])
        compressed = 4 * case["c_out"] * kk + 2 * kk * -(-case["c_out"] // case["tile"])
        return {"bytes": compressed + (4 * case["c_out"] * k if kind == "prune" else compressed), "flops": 0}
    if kind in ("net", "pointwise"):
        per_layer = [_conv_work(s, s.name.endswith("_c3") or (case.get("depth") in (18, 34) and s.name.endswith("_c2")))
                     for s in _layers(case)]
        pool = 0
        if kind == "net":
            stem, first = _layers(case)[:2]
            pool = 4 * (stem.pixels * stem.c_out + first.batch * first.h * first.w * first.c_in)
        return {"bytes": sum(b for b, _ in per_layer) + pool, "flops": sum(f for _, f in per_layer)}
    b, f = _conv_work(_layer(case), case["residual"])
    return {"bytes": b, "flops": f}


def tolerance(case):
    # pruning and the compressed form are exact: fp64 scores summed in one order, values copied
    if case["kind"] in ("prune", "import"):
        return "exact"
    # TF32 operands (10 explicit mantissa bits), fp32 sums; four times what comparison with fp64 convolutions of the same
    # pruned weights shows: 4.0e-4 for a layer, 3.2e-3 for a network's last map (it compounds its layers' rounding)
    return {"rel": 1.3e-2 if case["kind"] == "net" else 1.6e-3}
