"""What the library's speed is measured on: calls through its public entry points, as a user's program makes them.

A case is a dict of plain values:

    what      "forward"  fp_forward on images that are on the GPU
              "host"     fp_forward_host: pinned host images in, host logits out, waits
              "prune"    fp_prune at new ratios, the masks read back, and one fp_forward of the pruned network
              "soft"     one epoch of dynamic pruning (fp_soft_prune_epoch) and its masks read back
              "rank"     fp_rank_filters_static: score, rank and mask one filter bank
    net       resnet20/32/56/110 (CIFAR-shaped) or resnet18/34/50 (ImageNet-shaped), `hw` pixels high and wide
    batch     images of a forward
    ratios    what is pruned: "uniform" (`p` of every convolution), "drawn" (U(0.2, 0.6) per convolution), "inner" (`p` of
              the first two convolutions of every bottleneck block)
    dtype     of the images: "bf16" or "f32"
    graph     the forward replays a captured CUDA graph
    aggressive  the blocks are fused the paper's way (identity filters instead of an add) and pruned back
    norm      of the filter scores: "l1" or "l2"
    K, per    "rank": filters of the bank and weights per filter
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2010_16165_b200 import binding as fp
from paper_2010_16165_b200 import workloads as wl

CIFAR = {"resnet20": 3, "resnet32": 5, "resnet56": 9, "resnet110": 18}
BASIC = {"resnet18": (2, 2, 2, 2), "resnet34": (3, 4, 6, 3)}
NORMS = {"l1": fp.FP_NORM_L1, "l2": fp.FP_NORM_L2}


def _case(what, net, batch, ratios="uniform", p=0.3, hw=0, dtype="bf16", graph=True, aggressive=False, norm="l1"):
    return {"what": what, "net": net, "batch": batch, "ratios": ratios, "p": p, "hw": hw or (32 if net in CIFAR else 224),
            "dtype": dtype, "graph": graph, "aggressive": aggressive, "norm": norm}


def _rank_case(K, per, norm="l1"):
    return {"what": "rank", "K": K, "per": per, "p": 0.3, "norm": norm}


def listed():
    return [
        # the smallest call: one layer's bank ranked inside a program that must not allocate (64 filters of 64 x 3 x 3)
        dict(_rank_case(64, 576), name="rank_64x576"),
        # one 32 x 32 image at a time, as a device that answers single requests has it
        dict(_case("forward", "resnet20", 1, dtype="f32"), name="resnet20_b1_f32"),
        # a small batch of the smallest network with every option at its default (fp32 images, no graph)
        dict(_case("forward", "resnet20", 8, dtype="f32", graph=False), name="resnet20_b8_f32"),
        # CIFAR test-set evaluation and batched serving: the usual depth, and the deepest network at a large batch
        dict(_case("forward", "resnet56", 256), name="resnet56_b256"),
        dict(_case("forward", "resnet110", 1024, ratios="drawn"), name="resnet110_b1024"),
        # ImageNet-shaped serving batches: basic blocks, and the largest workload of all, bottleneck blocks
        dict(_case("forward", "resnet18", 64), name="resnet18_b64"),
        dict(_case("forward", "resnet50", 128, ratios="inner", p=0.4), name="resnet50_b128"),
        # single-image latency of the deep ImageNet-shaped network
        dict(_case("forward", "resnet50", 1, ratios="inner", p=0.4), name="resnet50_b1"),
        # a ragged batch of images of another size (50, 25, 13 and 7 pixels wide inside), fp32 as most decoders give them
        dict(_case("forward", "resnet34", 17, hw=200, dtype="f32"), name="resnet34_b17_hw200_f32"),
        # a request from host memory to host memory, the caller waiting for the answer
        dict(_case("host", "resnet18", 32), name="resnet18_b32_host"),
        # a search over pruning ratios: prune, read the masks, try the network
        dict(_case("prune", "resnet50", 8, ratios="inner", p=0.4, graph=False), name="resnet50_prune"),
        # Algorithm 1's loop: a trainer's update, then scores, masks and zeroed filters, once per epoch
        dict(_case("soft", "resnet50", 1, p=0.3, norm="l2"), name="resnet50_soft_epoch"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choices(["forward", "host", "prune", "soft", "rank"], [68, 8, 8, 8, 8])[0]
    if what == "rank":
        return _rank_case(_log_int(rng, 16, 2048), _log_int(rng, 3, 512) * rng.choice([1, 9, 9]), rng.choice(["l1", "l2"]))
    net = rng.choice(list(CIFAR) + ["resnet18", "resnet34", "resnet50"])
    c = _case(what, net, 1, norm=rng.choice(["l1", "l2"]))
    c["ratios"] = rng.choice(["uniform", "uniform", "drawn"] if net != "resnet50" else ["uniform", "inner", "inner"])
    c["p"] = 0.0 if rng.random() < 0.15 else round(rng.uniform(0.1, 0.6), 2)
    c["dtype"] = rng.choice(["bf16", "bf16", "f32"])
    c["graph"] = rng.random() < 0.6
    share = 0.8                                      # of the work of the largest listed case
    if net in CIFAR:
        c["aggressive"] = rng.random() < 0.12
        if rng.random() < 0.15:
            c["hw"], share = rng.choice([24, 28, 48, 64]), 0.01
        share = min(share, 0.2)
    elif rng.random() < 0.6:
        c["hw"] = 8 * rng.randint(16, 32)
        if rng.random() < 0.25:
            c["hw"], share = c["hw"] + rng.randint(-7, -1), 0.3
    if what in ("prune", "soft"):
        c["batch"], c["graph"] = _log_int(rng, 1, 16), False
        return c
    largest = max(work(x)["flops"] for x in listed() if x["what"] == "forward")
    most = int(share * largest / work(c)["flops"])
    c["batch"] = _log_int(rng, 1, max(1, min(most, 1024 if net in CIFAR else 256)))
    return c


def _net(case):
    net, hw = case["net"], case["hw"]
    if net in CIFAR:
        return wl.resnet_cifar(CIFAR[net], in_hw=hw, aggressive=case["aggressive"])
    if net in BASIC:
        return wl.resnet_imagenet_basic(BASIC[net], in_hw=hw)
    return wl.resnet_imagenet_bottleneck(in_hw=hw)


def _ratios(case, net, rng):
    if case["ratios"] == "inner":
        return wl.inner_bottleneck_ratios(case["p"])(net, rng)
    if case["ratios"] == "drawn":
        return wl.drawn_ratios(0.2, 0.6)(net, rng)
    return np.full(net.n_convs(), case["p"])


def _parameters(net, gen):
    """Weights and BN statistics of the repository's synthetic networks (workloads.make_params), drawn on the GPU."""
    w = torch.randn(net.n_weights, generator=gen, device="cuda")
    bn = torch.empty(net.n_bn, device="cuda")
    for n in net.nodes:
        if n["op"] == wl.OP_CONV:
            per = n["C"] * n["R"] * n["S"]
            w[n["w_off"]:n["w_off"] + n["K"] * per] *= math.sqrt(2.0 / per)
        elif n["op"] == wl.OP_FC:
            w[n["w_off"]:n["w_off"] + n["K"] * n["C"]] *= math.sqrt(2.0 / n["C"])
            w[n["b_off"]:n["b_off"] + n["K"]] = 0.0
        elif n["op"] == wl.OP_BN:
            gamma, beta, mean, var = bn[n["bn_off"]:n["bn_off"] + 4 * n["K"]].view(4, n["K"])
            gamma.uniform_(0.5, 1.5, generator=gen)
            beta.normal_(0.0, 0.1, generator=gen)
            mean.normal_(0.0, 0.1, generator=gen)
            var.uniform_(0.5, 1.5, generator=gen)
    return w, bn


_one_stream = []


def _stream():
    """The stream a program runs its network on (one for all states: passes follow one another)."""
    if not _one_stream:
        _one_stream.append(torch.cuda.Stream())
    return _one_stream[0]


class _State:
    handle = None

    def __del__(self):
        if self.handle is not None:
            fp.fp_destroy(self.handle)


def prepare(case, seed):
    s = _State()
    s.what, s.stream = case["what"], _stream()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    s.norm = NORMS[case["norm"]]
    if s.what == "rank":
        s.K, s.per = case["K"], case["per"]
        s.q = int(case["p"] * s.K)
        s.bank = torch.randn(s.K * s.per, generator=gen, device="cuda") * math.sqrt(2.0 / s.per)
        s.rank = torch.empty(s.K, dtype=torch.int32, device="cuda")
        s.mask = torch.empty(s.K, dtype=torch.uint8, device="cuda")
        return s
    net = _net(case)
    w, bn = _parameters(net, gen)
    s.batch = case["batch"]
    s.ratios = _ratios(case, net, np.random.default_rng(seed))
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s.handle = fp.fp_fuse(net, w, bn, s.batch, in_dtype=fp.FP_DTYPE_BF16 if case["dtype"] == "bf16" else fp.FP_DTYPE_F32,
                          use_graph=int(case["graph"]))
    if s.what == "soft":
        # a trainer's step: a hundredth of a weight's standard deviation per epoch, every convolution in order
        convs = [n for n in net.nodes if n["op"] == wl.OP_CONV]
        elems = fp.conv_bank_elems(s.handle)
        s.updates = torch.randn(sum(elems), generator=gen, device="cuda") * 0.01
        off = 0
        for n, count in zip(convs, elems):
            s.updates[off:off + count] *= math.sqrt(2.0 / (n["C"] * n["R"] * n["S"]))
            off += count
        return s
    s.images = torch.randn(s.batch, 3, case["hw"], case["hw"], generator=gen, device="cuda").to(dtype)
    if s.what == "host":
        s.images = s.images.cpu().pin_memory()
    s.logits = torch.empty(s.batch, net.n_classes(), device="cpu" if s.what == "host" else "cuda", pin_memory=s.what == "host")
    if s.what != "prune":
        fp.fp_prune(s.handle, s.ratios, norm=s.norm)
    return s


def _masks(handle):
    got = [v for v in fp.masks_and_ranks(handle).values() if v[0] is not None]
    return np.concatenate([m for m, _ in got]), np.concatenate([r for _, r in got])


def run(s):
    if s.what == "forward":
        fp.fp_forward(s.handle, s.images, s.batch, s.logits, s.stream)
        return s.logits
    if s.what == "host":
        fp.fp_forward_host(s.handle, s.images, s.batch, s.logits, s.stream)
        return s.logits
    if s.what == "prune":
        fp.fp_prune(s.handle, s.ratios, norm=s.norm)
        masks, ranks = _masks(s.handle)
        fp.fp_forward(s.handle, s.images, s.batch, s.logits, s.stream)
        return {"masks": masks, "ranks": ranks, "logits": s.logits}
    if s.what == "soft":
        fp.fp_soft_prune_epoch(s.handle, s.ratios, s.updates, norm=s.norm)
        masks, ranks = _masks(s.handle)
        return {"masks": masks, "ranks": ranks}
    fp.fp_rank_filters_static(s.bank, s.K, s.per, s.norm, s.q, s.rank, s.mask, s.stream)
    return {"rank": s.rank, "mask": s.mask}


def _sizes(case):
    """(flops per image, kept weights, all convolution weights, all filters, FC weights) of the network after pruning: removed
    filters cost nothing, nor do the input channels they fed where every reader is a convolution."""
    net = _net(dict(case, aggressive=False))
    ratios = _ratios(case, net, np.random.default_rng(0)) if not case["aggressive"] else np.zeros(net.n_convs())
    readers = {}
    for n in net.nodes:
        for src in (n["in0"], n["in1"] if n["op"] == wl.OP_ADD else -1):
            if src >= 0:
                readers.setdefault(src, []).append(n["op"])
    kept = {-1: net.in_C}                 # channels of every node's output that are left
    size = {-1: case["hw"]}
    made_by_conv = {-1: False}            # a convolution's output, or that behind BN, ReLU and pooling
    full = {-1: net.in_C}
    flops = weights = every = filters = fc = 0
    conv = 0
    for i, n in enumerate(net.nodes):
        src = n["in0"]
        hw, ch = size[src], kept[src] if made_by_conv[src] else full[src]
        full[i] = full[src] if n["op"] in (wl.OP_RELU, wl.OP_ADD) else n["K"]
        made_by_conv[i] = made_by_conv[src] and n["op"] != wl.OP_ADD and wl.OP_ADD not in readers.get(i, [])
        kept[i], size[i] = ch, hw
        if n["op"] == wl.OP_CONV:
            k = n["K"] - int(math.floor(ratios[conv] * n["K"] + 1e-9))
            conv += 1
            size[i] = (hw + 2 * n["pad"] - n["R"]) // n["stride"] + 1
            kept[i], made_by_conv[i] = k, True
            flops += 2 * size[i] ** 2 * k * ch * n["R"] * n["S"]
            weights += k * ch * n["R"] * n["S"]
            every += n["K"] * n["C"] * n["R"] * n["S"]
            filters += n["K"]
        elif n["op"] == wl.OP_MAXPOOL:
            size[i] = (hw + 2 * n["pad"] - n["R"]) // n["stride"] + 1
        elif n["op"] == wl.OP_SHORTCUT_A:
            size[i], made_by_conv[i] = -(-hw // n["stride"]), False
        elif n["op"] == wl.OP_FC:
            flops += 2 * n["K"] * n["C"]
            fc += n["K"] * n["C"]
    return flops, weights, every, filters, fc


def work(case):
    if case["what"] == "rank":
        return {"bytes": 4 * case["K"] * case["per"] + 5 * case["K"], "flops": 2 * case["K"] * case["per"]}
    flops, weights, every, filters, fc = _sizes(case)
    images = case["batch"] * 3 * case["hw"] ** 2 * (2 if case["dtype"] == "bf16" else 4)
    logits = 4 * case["batch"] * (10 if case["net"] in CIFAR else 1000)
    forward = {"bytes": images + 2 * weights + 4 * fc + logits, "flops": flops * case["batch"]}
    if case["what"] == "prune":           # every fused weight is read to score it, the packed filters are written, the forward reads them
        return {"bytes": 4 * every + 2 * weights + 5 * filters + forward["bytes"], "flops": 2 * every + forward["flops"]}
    if case["what"] == "soft":            # weights and updates read, updated weights written
        return {"bytes": 12 * every + 5 * filters, "flops": 3 * every}
    return forward


def tolerance(case):
    if case["what"] in ("rank", "soft"):  # scores have one defined summation order in fp64: masks and ranks are one answer
        return "exact"
    # every layer rounds its filters and its output to bf16, and a network averages the layers' roundings: two correct
    # orders of summation differ by about that on the logits of a network tens of layers deep
    return {"rel": 1e-2, "max": 5e-2}
