"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is one pass through the public entry points of `paper_2503_20354_b200.binding`, on inputs
and buffers that such a program has in hand.  There are three kinds:

  step        one adaptation step over some blocks of a network: the ratio rule (Eq. 5-7) over the
              whole network, prune+compact of every saved activation (the forward pass), then the
              weight gradients in reverse order (the backward pass)
  importance  the pass that measures Gradient Importance: the same at one static ratio, then Eq. 4
              for every layer, a host read of the G_i and the ratio rule on them
  tensor      one activation tensor pruned and stored, and in some cases rebuilt

`listed()` gives the fixed cases, `draw(rng)` one more of the same ranges.
"""
from __future__ import annotations

import math

import torch

from paper_2503_20354_b200 import binding as B
from paper_2503_20354_b200 import workloads as W

# output-gradient scale per network (as the benchmark has it)
SIGMA = {"tiny": 0.01, "wrn28": 0.01, "resnext29": 0.01, "segformer": 0.01, "resnet50": 1e-3, "vit": 1e-3}
# the batch the paper adapts each network at: the largest a case takes
FULL_BATCH = {"tiny": 16, "wrn28": 200, "resnext29": 200, "segformer": 1, "resnet50": 64, "vit": 64}
BLOCKS = {
    "wrn28": ["conv1"] + ["g%db%d" % (g, b) for g in (1, 2, 3) for b in range(4)],
    "resnext29": ["conv1"] + ["s%db%d" % (s, b) for s in (1, 2, 3) for b in range(3)] + ["fc"],
    "resnet50": ["stem"] + ["layer%d.%d" % (s + 1, b) for s, k in enumerate((3, 4, 6, 3)) for b in range(k)] + ["fc"],
    "segformer": ["s%db%d" % (s, b) for s, k in enumerate((3, 6, 40, 3)) for b in range(k)],
    "vit": ["blk%d" % b for b in range(12)],
}


def _step(name, net, blocks, batch, ratios="rule", path=B.PATH_TENSOR_CORE, drop_zeros=False, streams=1,
          image=0, own_buffers=True, kind="step"):
    return {"name": name, "kind": kind, "net": net, "blocks": blocks, "batch": batch, "ratios": ratios,
            "path": path, "drop_zeros": drop_zeros, "streams": streams, "image": image,
            "own_buffers": own_buffers}


def _tensor(name, n, dtype, dist, ratio, drop_zeros=False, rebuild=False, static=False):
    return {"name": name, "kind": "tensor", "n": n, "dtype": dtype, "dist": dist, "ratio": ratio,
            "drop_zeros": drop_zeros, "rebuild": rebuild, "static": static}


def listed():
    return [
        # one small 3x3 convolution, everything but its inputs left to the call: what a first user tries
        _step("tiny conv", "tiny", "", 16, ratios="0.6", own_buffers=False),
        # a transformer block at the benchmark's batch: bf16 activations, four linear layers
        _step("vit block", "vit", "blk3", 64),
        # one residual block of each width of WideResNet-28-10 at the paper's batch: fp32 activations,
        # 3x3 convolutions at 32x32, 16x16 and 8x8, a strided one and its shortcut
        _step("wrn blocks", "wrn28", "g1b1,g2b0,g3b1", 200),
        # ResNet-50's stem and first blocks: the large maps, 7x7 and strided convolutions
        _step("resnet early", "resnet50", "stem,layer1.0,layer2.0", 64, ratios="uniform"),
        # its deep blocks (14x14 and 7x7 maps) and the classifier, the layers issued on eight streams
        # as the benchmark does
        _step("resnet late, 8 streams", "resnet50", "layer3.1,layer4.0,fc", 64, streams=8),
        # ResNeXt-29's grouped convolutions, the stores without the zeros that ReLU leaves
        _step("resnext blocks", "resnext29", "s1b0,s2b0,s3b2", 200, drop_zeros=True),
        # segmentation at batch 1: many small calls (linear, reduction and depthwise layers)
        _step("segformer block", "segformer", "s2b4", 1, image=1024),
        # a user who wants fp32 products: the CUDA-core path
        _step("fp32 path", "wrn28", "g2b1", 16, path=B.PATH_FP32),
        # the importance pass of Algorithm 1 at its static ratio, at a small online batch
        _step("importance pass", "wrn28", "conv1,g1b0,g2b1,g3b1", 24, ratios="0.9", kind="importance"),
        # a small ragged tensor from a caller that cannot allocate, with many equal magnitudes
        _tensor("small ties", 1000003, "bf16", "ties16", 0.9, static=True),
        # an activation cached and rebuilt (layers whose weight gradient the user computes densely)
        _tensor("cache and rebuild", 64 * 197 * 3072 + 77, "bf16", "gelu_normal", 0.7, rebuild=True),
        # the largest tensor of the bandwidth sweep
        _tensor("largest tensor", 1 << 30, "fp32", "relu_normal", 0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "tensor", "tensor", "importance"])
    if kind == "tensor":
        n = _log_int(rng, 1 << 17, 1 << 28) | rng.randrange(2)
        dist = rng.choice(["relu_normal", "normal", "student_t2", "gelu_normal", "ties16"])
        c = _tensor("", n, rng.choice(["fp32", "bf16"]), dist, round(rng.uniform(0.1, 0.99), 3),
                    drop_zeros=dist == "relu_normal" and rng.random() < 0.4)
        c["rebuild"] = rng.random() < 0.3
        c["static"] = n <= B.SURGEON_STATIC_MAX_N and not c["drop_zeros"] and rng.random() < 0.4
    else:
        net = rng.choice(["tiny", "wrn28", "resnet50", "vit", "resnext29", "segformer"])
        blocks = "" if net == "tiny" else ",".join(sorted(rng.sample(BLOCKS[net], 1 if net in ("vit", "segformer") else 2)))
        c = _step("", net, blocks, _log_int(rng, 1, FULL_BATCH[net]), kind=kind)
        c["image"] = 32 * rng.randint(8, 32) if net == "segformer" else 0
        if kind == "importance":
            c["ratios"] = "0.9"
        else:
            c["ratios"] = rng.choice(["rule", "uniform", "%.2f" % rng.uniform(0.0, 0.95)])
            c["drop_zeros"] = rng.random() < 0.25
            c["streams"] = rng.choice([1, 1, 1, 8])
            c["own_buffers"] = c["streams"] > 1 or c["ratios"] in ("rule", "uniform") or rng.random() < 0.5
            if rng.random() < 0.15:             # the fp32 path, kept to sizes that one would use it at
                c["path"], c["image"] = B.PATH_FP32, min(c["image"], 512)
                c["batch"] = max(1, min(c["batch"], int(c["batch"] * 3e10 / sum(l.flops for l in _layers(c)[0]))))
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------------------------

def _network(case):
    b = case["batch"]
    if case["net"] == "segformer":
        return W.segformer_b5(case["image"], b)
    return {"tiny": W.tiny_conv, "wrn28": W.wrn28_10, "resnet50": W.resnet50, "vit": W.vit_b16,
            "resnext29": W.resnext29}[case["net"]](b)


def _layers(case):
    """(layers of the case's blocks, their places in the network, the network)."""
    net = _network(case)
    want = case["blocks"].split(",")
    at = [i for i, l in enumerate(net)
          if case["net"] == "tiny" or l.name in want or l.name.rsplit(".", 1)[0] in want]
    return [net[i] for i in at], at, net


def _ratios(case, seed, net):
    """Ratios of all layers of the network."""
    if case["ratios"] == "rule":
        gi = W.gradient_importance(len(net), seed)
        return B.surgeon_layer_ratios(gi, [l.act_bytes for l in net], allow_degenerate=True)
    if case["ratios"] == "uniform":
        return W.uniform_ratios(len(net), seed)
    return [float(case["ratios"])] * len(net)


def _bits(values):
    return values.view(torch.int32 if values.dtype == torch.float32 else torch.int16)


class _StepState:
    def __init__(self, case, seed):
        dev = torch.device("cuda")
        layers, at, net = _layers(case)
        self.case, self.at, self.n_net = case, at, len(net)
        self.gi = W.gradient_importance(len(net), seed)
        self.lam = [float(l.act_bytes) for l in net]
        ratios = list(_ratios(case, seed, net))
        # layers that read one tensor share its store, pruned at the smaller of their ratios
        self.shared = W.shared_inputs(layers)
        self.own = [j for j in range(len(layers)) if j not in self.shared]
        self.least = [[at[j]] for j in range(len(layers))]
        for j, i in self.shared.items():
            self.least[i].append(at[j])
        self.static = None if case["ratios"] == "rule" else ratios
        self.flags = B.SURGEON_STORE_DROP_ZEROS if case["drop_zeros"] else 0
        self.desc = [B.layer_desc(l, case["path"]) for l in layers]
        self.x = {j: W.activation(layers[j], seed, at[j], device=dev) for j in self.own}
        self.g = [W.grad_out(l, seed, at[j], sigma=SIGMA[case["net"]], device=dev) for j, l in enumerate(layers)]
        self.streams = [torch.cuda.Stream() for _ in range(case["streams"])] if case["streams"] > 1 else [None]
        self.dw = self.store = self.out = None
        self.ws = [None] * len(self.streams)
        if case["own_buffers"]:
            self.dw = [torch.empty(l.dw_shape, device=dev) for l in layers]
            # sized for ratio 0: ratios change every batch, the buffers do not (a call leaves the end of
            # a buffer that no value reaches as it is)
            self.store = {j: B.CompressedActivation(layers[j].n_act, layers[j].dt, 0.0, dev) for j in self.own}
            for s in self.store.values():
                s.values.zero_()
            need = max([s.sizes.workspace_bytes for s in self.store.values()]
                       + [B.surgeon_weight_grad_workspace(d) for d in self.desc] + [256])
            self.ws = [torch.empty(need, dtype=torch.uint8, device=dev) for _ in self.streams]
            self.out = [[s.bitmap, _bits(s.values), s.block_offsets, s.header] for s in self.store.values()]
        if case["kind"] == "importance":
            self.g_i = torch.zeros(len(layers), dtype=torch.float64, device=dev)
            self.g_at = [self.g_i[j:j + 1] for j in range(len(layers))]


class _TensorState:
    def __init__(self, case, seed):
        dev = torch.device("cuda")
        self.case = case
        x = W.draw(case["dist"], case["n"], seed, 0, device=dev)
        self.x = x if case["dtype"] == "fp32" else x.to(torch.bfloat16)
        self.flags = B.SURGEON_STORE_DROP_ZEROS if case["drop_zeros"] else 0
        self.store = B.CompressedActivation(case["n"], B.dtype_code(self.x.dtype), case["ratio"], dev)
        self.store.values.zero_()
        self.ws = torch.empty(self.store.sizes.workspace_bytes, dtype=torch.uint8, device=dev)
        s = self.store
        self.out = [s.bitmap, _bits(s.values), s.block_offsets, s.header]


def prepare(case, seed):
    return _TensorState(case, seed) if case["kind"] == "tensor" else _StepState(case, seed)


# ---- one pass ---------------------------------------------------------------------------------

def _run_tensor(s):
    c = s.case
    if c["static"]:
        B.surgeon_prune_compact_static(s.x, c["ratio"], s.store)
    else:
        B.surgeon_prune_compact(s.x, c["ratio"], out=s.store, workspace=s.ws, flags=s.flags)
    return s.out + [B.surgeon_decompress(s.store)] if c["rebuild"] else s.out


def _run_step(s):
    ratios = s.static
    if ratios is None:
        ratios = B.surgeon_layer_ratios(s.gi, s.lam, allow_degenerate=True)
    many = len(s.streams)
    main = torch.cuda.current_stream()
    if many > 1:
        for st in s.streams:
            st.wait_stream(main)
    store, out = s.store, s.out
    if store is None:
        store = {j: B.surgeon_prune_compact(s.x[j], min(ratios[i] for i in s.least[j]), flags=s.flags) for j in s.own}
        # (the end of a fresh buffer that no value reaches is not the call's)
        out = [[v.bitmap, v.block_offsets, v.header] + ([] if s.flags else [_bits(v.values)]) for v in store.values()]
    else:
        for j in s.own:
            B.surgeon_prune_compact(s.x[j], min(ratios[i] for i in s.least[j]), out=store[j],
                                    workspace=s.ws[j % many], stream=s.streams[j % many], flags=s.flags)
    if many > 1:
        for st in s.streams:
            main.wait_stream(st)
        for st in s.streams:
            st.wait_stream(main)
    dw = [None] * len(s.desc)
    for j in reversed(range(len(s.desc))):
        dw[j] = B.surgeon_weight_grad(store[s.shared.get(j, j)], s.desc[j], s.g[j], dw=s.dw[j] if s.dw else None,
                                      workspace=s.ws[j % many], stream=s.streams[j % many])
    if many > 1:
        for st in s.streams:
            main.wait_stream(st)
    if s.case["kind"] != "importance":
        return out, dw
    for j, d in enumerate(dw):
        B.surgeon_gradient_importance(d, out=s.g_at[j], workspace=s.ws[0])
    gi = s.g_i.cpu().numpy()
    return out, dw, gi, B.surgeon_layer_ratios(gi, [s.lam[i] for i in s.at], allow_degenerate=True)


def run(state):
    return _run_tensor(state) if state.case["kind"] == "tensor" else _run_step(state)


# ---- what a pass cannot do without ------------------------------------------------------------

def _store_bytes(n, dt, ratio):
    s = B.surgeon_compact_sizes(n, dt, ratio)
    return s.bitmap_bytes + s.values_bytes + s.offsets_bytes


def work(case):
    if case["kind"] == "tensor":
        dt = B.SURGEON_F32 if case["dtype"] == "fp32" else B.SURGEON_BF16
        dense = case["n"] * (4 if dt == B.SURGEON_F32 else 2)
        return {"bytes": (dense + _store_bytes(case["n"], dt, case["ratio"])) * (2 if case["rebuild"] else 1), "flops": 0}
    layers, at, net = _layers(case)
    ratios = _ratios(case, 1, net)
    shared = W.shared_inputs(layers)
    total = 0
    for j, l in enumerate(layers):
        store = _store_bytes(l.n_act, l.dt, float(ratios[at[j]]))
        if j not in shared:
            total += l.act_bytes + store                       # read the activation, write the store
        total += store + 4 * math.prod(l.grad_shape) + 4 * l.n_weight   # read both operands, write dW
    return {"bytes": total, "flops": sum(l.flops for l in layers)}


def tolerance(case):
    """Stores (returned as whole numbers) are the same to the last bit.  Weight gradients: sums of
    up to 10^5 products in fp32, whose order differs; the tensor-core path rounds its operands to
    bf16 first, the same way in any implementation, so it is the sum that differs there too."""
    if case["kind"] == "tensor":
        return "exact"
    return {"rel": 1e-5, "max": 1e-3} if case["path"] == B.PATH_FP32 else {"rel": 5e-4, "max": 2e-2}
