"""What the performance of this framework is measured on: training and inference of the residual networks it
exists for, through the entry points of `paper_1906_09108_b200.binding`.

A training case is a run in flight: the pipeline of K modules is full and (with graphs) every phase of the rings is
recorded.  One pass is one logging interval of a training loop: `steps` iterations on the next batches of a pool,
each with its loss kept, then the wait that ends an interval, then the state a program reads there -- every module's
parameters and running batch-norm statistics, into buffers on the GPU.  The pool (16 batches) stands for a data
loader; `feed` says whether the loader hands over GPU tensors or pinned host buffers.

An inference case is a test set summed over batches: `steps` calls of `eval`, each with its logits kept and the
top-1 matches added up on the GPU.

Learning rate 0.01 everywhere: the warm-up rate such runs begin with.  Images are normal, labels uniform, weights
He-normal with batch-norm scales and shifts spread around 1 and 0.
"""
import math

import torch

from paper_1906_09108_b200 import binding as B

POOL = 16

# Networks by name: everything about the architecture but the batch.
_6N2 = dict(family="resnet6n2", widths=(16, 32, 64), stem_width=16, in_h=32, in_w=32, classes=10)
_NETS = {
    "tiny": dict(_6N2, blocks=(1, 1, 1), widths=(8, 16, 32), stem_width=8, in_h=16, in_w=16),
    "resnet20": dict(_6N2, blocks=(3, 3, 3)),
    "resnet56": dict(_6N2, blocks=(9, 9, 9)),
    "resnet110": dict(_6N2, blocks=(18, 18, 18)),
    "resnet1202": dict(_6N2, blocks=(200, 200, 200)),
    "resnet18": dict(_6N2, blocks=(2, 2, 2, 2), widths=(64, 128, 256, 512), stem_width=64),
    "wrn28_10": dict(family="wrn", blocks=(4, 4, 4), widths=(160, 320, 640), stem_width=16, in_h=32, in_w=32, classes=100),
}
_NETS["wrn16_4"] = dict(_NETS["wrn28_10"], blocks=(2, 2, 2), widths=(64, 128, 256))


def _case(name, net, **kw):
    c = dict(mode="train", batch=128, K=2, precision="bf16", graphs=True, feed="device", order="backward_first",
             weights="stashed", shortcut="projection", beta=0.5, steps=8)
    c.update(net if isinstance(net, dict) else _NETS[net])
    c.update(kw)
    blocks, widths = c["blocks"], c["widths"]
    c["blocks"], c["widths"] = ",".join(map(str, blocks)), ",".join(map(str, widths))
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run there is a configuration for: what an iteration costs when the kernels cost nothing
        _case("tiny_k2", "tiny", batch=8, beta=0.2, steps=16),
        # a small network with the constructor's defaults for issuing (streams, no graphs): the host launches every kernel
        _case("resnet20_k2_streams", "resnet20", beta=0.2, graphs=False),
        # the exact mode (fp32 storage and arithmetic), the constructor's default precision, as reference runs use it
        _case("resnet20_k2_fp32", "resnet20", beta=0.2, precision="fp32"),
        _case("resnet56_k2", "resnet56"),
        # three modules, forward-first schedule, zero-padded shortcuts, a batch and an image size that fill no tile
        _case("resnet56_k3_ragged", "resnet56", K=3, batch=97, in_h=28, in_w=28, beta=0.3, order="forward_first",
              shortcut="zero_pad"),
        # the benchmark's network, fed from pinned host memory as a training program feeds it
        _case("resnet110_k4_host", "resnet110", K=4, beta=0.2, feed="host"),
        # the deepest network of the tables, on the batch that its configuration has
        _case("resnet1202_k4", "resnet1202", K=4, batch=64, steps=4),
        # wide layers: four stages to 512 channels, and the wide residual network with 100 classes
        _case("resnet18_k2", "resnet18"),
        _case("wrn28_10_k2", "wrn28_10", beta=0.6),
        # a small wide network on 24x24 crops, whose maps (24, 12, 6) are no power of two
        _case("wrn16_4_crop24", "wrn16_4", in_h=24, in_w=24, beta=0.6),
        # test sets: the deep narrow network and the wide one
        _case("resnet110_eval", "resnet110", K=4, mode="eval"),
        _case("wrn28_10_eval", "wrn28_10", mode="eval", steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Networks of the same families between the listed ones: depth, width, batch, image size, K and options."""
    kind = rng.choice(("narrow", "narrow", "narrow", "wide4", "wrn"))
    mode = rng.choice(("train", "train", "train", "train", "eval"))
    batch = _log_int(rng, 8, 160)
    sizes = (16, 32, 32)
    precision = "bf16"
    if kind == "narrow":
        precision = rng.choice(("bf16", "bf16", "bf16", "fp32"))
        base = rng.choice((8, 16, 16, 16, 24, 32))
        deepest = {24: 3, 32: 9}.get(base, 30)
        if precision == "fp32":              # the exact mode is for small runs
            base, deepest = min(base, 16), 4
        n = _log_int(rng, 1, deepest)
        blocks, widths = (n,) * 3, (base, 2 * base, 4 * base)
        net = dict(_6N2, stem_width=base)
        sizes = (16, 24, 28, 32, 32, 40)
    elif kind == "wide4":
        n = rng.randint(1, 3)
        base = rng.choice((32, 48, 64))
        sizes += (24,) if base == 32 else ()
        blocks, widths = (n,) * 4, (base, 2 * base, 4 * base, 8 * base)
        net = dict(_6N2, stem_width=base)
    else:
        n = rng.randint(1, 4)
        base = 16 * rng.randint(2, 10)
        sizes += (24,) if n <= 2 and base <= 64 else ()
        blocks, widths = (n,) * 3, (base, 2 * base, 4 * base)
        net = dict(_NETS["wrn28_10"])
        batch = min(batch, 128)
    net["blocks"], net["widths"] = blocks, widths
    net["in_h"] = net["in_w"] = rng.choice(sizes)
    net["classes"] = rng.choice((10, 100, rng.randint(2, 200)))
    return _case(None, net, mode=mode, batch=batch, K=min(rng.choice((1, 2, 2, 3, 4)), sum(blocks)), precision=precision,
                 graphs=rng.random() < 0.75, feed=rng.choice(("device", "device", "host")),
                 order=rng.choice(("backward_first", "backward_first", "forward_first")),
                 weights=rng.choice(("stashed", "stashed", "stashed", "current")),
                 shortcut=rng.choice(("projection", "projection", "zero_pad")) if kind == "narrow" else "projection",
                 beta=rng.choice((0.2, 0.5, 0.6, 1.0)), steps=rng.choice((4, 5, 8)))


def _lists(case):
    return [int(v) for v in case["blocks"].split(",")], [int(v) for v in case["widths"].split(",")]


def _splits(case):
    """Module ends: the blocks divided as evenly as they can be, as the configurations do."""
    nb = sum(_lists(case)[0])
    return tuple(round(nb * (i + 1) / case["K"]) for i in range(case["K"] - 1))


def _ok(g, status):
    if status != B.FDG_OK:
        raise B.FDGError(status, g.lib.fdg_last_error(g.ctx).decode())


def _init_params(layout, gen, depth):
    """One module's parameters in flat order.  The scale of a post-activation block's second batch norm is divided by
    the square root of the number of blocks: the residual branches of a network that trains are that small, and a deep
    network's gradients neither explode nor hang on the last bit of its first layers."""
    parts = []
    bound = 1.0
    unit, gammas = None, 0
    for name, kind, shape in layout:
        n = math.prod(shape)
        if name.split("@")[0] != unit:
            unit, gammas = name.split("@")[0], 0
        if kind == "conv":
            p = torch.randn(n, device="cuda", generator=gen) * math.sqrt(2.0 / math.prod(shape[1:]))
        elif kind == "bn_gamma":
            p = torch.rand(n, device="cuda", generator=gen) + 0.5
            gammas += 1
            if depth and unit.startswith("block") and gammas == 2:
                p /= math.sqrt(depth)
        elif kind == "bn_beta":
            p = torch.randn(n, device="cuda", generator=gen) * 0.1
        else:
            if kind == "fc_w":
                bound = 1.0 / math.sqrt(shape[1])
            p = (torch.rand(n, device="cuda", generator=gen) * 2 - 1) * bound
        parts.append(p)
    return torch.cat(parts)


def prepare(case, seed):
    blocks, widths = _lists(case)
    arch = B.make_arch(family=case["family"], blocks=blocks, widths=widths, stem_width=case["stem_width"], in_h=case["in_h"],
                       in_w=case["in_w"], in_c=3, num_classes=case["classes"], batch=case["batch"], shortcut=case["shortcut"])
    train = case["mode"] == "train"
    g = B.FDG(arch, K=case["K"], split_after_block=_splits(case), beta=case["beta"], lr=0.01 if train else 0.0,
              weight_decay=5e-4 if train else 0.0, graphs=case["graphs"],
              order=B.FDG_FORWARD_FIRST if case["order"] == "forward_first" else B.FDG_BACKWARD_FIRST,
              weight_reading=B.FDG_CURRENT if case["weights"] == "current" else B.FDG_STASHED,
              precision=B.FDG_BF16_TC if case["precision"] == "bf16" else B.FDG_FP32_CUDACORE)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    for k in range(1, case["K"] + 1):
        p = _init_params(g.param_layout(k), gen, sum(blocks) if case["family"] == "resnet6n2" else 0)
        _ok(g, g.lib.fdg_set_params(g.ctx, k, p.data_ptr(), p.numel()))
    shape = (case["batch"], case["in_h"], case["in_w"], 3)
    pool = []
    for _ in range(POOL):
        x = torch.randn(shape, device="cuda", generator=gen)
        y = torch.randint(0, case["classes"], (case["batch"],), device="cuda", generator=gen, dtype=torch.int32)
        pool.append((x, y))
    # the pipeline filled and every phase of the rings met once; for inference this is what gives the running
    # statistics their values (the learning rate is 0 there: the weights stay)
    for i in range(2 * case["K"] + 14):
        g.step(*pool[i % POOL])
    g.sync()
    state = dict(g=g, train=train, host=case["feed"] == "host", steps=case["steps"], at=0)
    if not train:
        state["logits"] = torch.empty((case["steps"], case["batch"], case["classes"]), device="cuda")
    elif state["host"]:
        pool = [(x.cpu().pin_memory(), y.cpu().pin_memory()) for x, y in pool]
        state["loss"] = torch.zeros(case["steps"]).pin_memory()
    else:
        state["loss"] = torch.zeros(case["steps"], device="cuda")
    state["pool"] = pool
    if train:
        n = B.C.c_size_t()
        state["params"], state["running"] = [], []
        for k in range(1, case["K"] + 1):
            state["params"].append(torch.empty(g.param_count(k), device="cuda"))
            _ok(g, g.lib.fdg_bn_running_count(g.ctx, k, B.C.byref(n)))
            state["running"].append(torch.empty(n.value, device="cuda"))
    torch.cuda.synchronize()
    return state


def run(state):
    g, steps, pool = state["g"], state["steps"], state["pool"]
    at = state["at"]
    state["at"] = at + steps
    if not state["train"]:
        correct = torch.zeros(1, dtype=torch.int32, device="cuda")
        for i in range(steps):
            x, y = pool[i]
            g.eval(x, y, logits_dev=state["logits"][i], correct_dev=correct)
        return {"logits": state["logits"]}       # the count hangs on ties within rounding: the logits hold it
    step = g.step_host if state["host"] else g.step
    for i in range(steps):
        x, y = pool[(at + i) % POOL]
        step(x, y, state["loss"][i:i + 1])
    g.sync()
    for k, (p, r) in enumerate(zip(state["params"], state["running"]), 1):
        _ok(g, g.lib.fdg_get_params(g.ctx, k, p.data_ptr(), p.numel()))
        if r.numel():
            _ok(g, g.lib.fdg_get_bn_running(g.ctx, k, r.data_ptr(), r.numel()))
    return {"loss": state["loss"], "params": state["params"], "running": state["running"]}


def _counts(case):
    """Per image: multiply-adds of the forward pass (and those of the stem), elements of all convolution outputs;
    parameters."""
    blocks, widths = _lists(case)
    h, w, ci = case["in_h"], case["in_w"], case["stem_width"]
    stem = h * w * ci * 27
    macs, acts, params = stem, h * w * ci, 27 * ci + 2 * ci
    for s, (n, co) in enumerate(zip(blocks, widths)):
        for b in range(n):
            stride = 2 if s > 0 and b == 0 else 1
            h, w = h // stride, w // stride
            proj = (stride != 1 or ci != co) and case["shortcut"] == "projection"
            wts = 9 * ci * co + 9 * co * co + (ci * co if proj else 0)
            macs += h * w * wts
            acts += h * w * co * (3 if proj else 2)
            params += wts + 4 * co
            ci = co
    return macs + ci * case["classes"], stem, acts, params + (ci + 1) * case["classes"]


def work(case):
    """Training: forward, data gradient (not of the images) and weight gradient of every convolution; every
    convolution's output written once and read once (a batch norm needs all of it, and the delayed backward comes
    iterations later); images, parameters and momentum.  Inference: images, parameters, logits; the forward pass."""
    macs, stem, acts, params = _counts(case)
    b, t = case["batch"], case["steps"]
    size = 2 if case["precision"] == "bf16" else 4
    image = case["in_h"] * case["in_w"] * 3 * 4
    if case["mode"] == "eval":
        return {"flops": 2.0 * macs * b * t, "bytes": float(t * b * (image + 4 * case["classes"]) + 4 * params)}
    return {"flops": 2.0 * (3 * macs - stem) * b * t, "bytes": float(t * (b * (image + 2 * acts * size) + 16 * params))}


def tolerance(case):
    """Tensors between two layers are kept in bf16 in the bf16 mode.  A sum taken in another order moves some of them
    by one rounding step, which moves a few ReLU gates, and the gradients behind those; iterations of training add up.
    (The same run with the images of every batch in another order, which changes nothing but the order of sums:
    up to 8e-3 in bf16, 4e-6 in fp32.)"""
    if case["precision"] == "fp32":
        return {"rel": 5e-5, "max": 2e-3}
    return {"rel": 0.015, "max": 0.25}
