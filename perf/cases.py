"""Timed cases: what a program does with this library, through its public calls.

A case is one pass over buffers the program keeps (packed filters, BatchNorm vectors, scratch):

  block   BatchNorm -> BinActiv -> BinConv of one layer, with the options of the block: residual
          (ResNet shortcut), ReLU, max pooling, border variant of K, and `weights`: the real filters
          are binarised in the same pass, as in a training step (at inference they are kept packed)
  kbit    the block with k-bit activations
  bwn     the Binary-Weight-Network convolution: real inputs, +-1 filters
  bgrad   the backward convolution with a binarised gradient; filters packed in the same pass
  chain   the 16 binary layers of ResNet-18 with their shortcuts (runner.ChainRunner)
"""
import math

import torch

import paper_1603_05279_b200 as X
from paper_1603_05279_b200 import workloads as wl
from paper_1603_05279_b200.runner import ChainRunner


def _layer(name, kind, N, C, H, W, Co, k, stride, pad, **more):
    c = {"name": name, "kind": kind, "N": N, "C": C, "H": H, "W": W, "Co": Co, "k": k,
         "stride": stride, "pad": pad, "w_std": 1.0}
    c.update(more)
    return c


def listed():
    return [
        # one image through one small layer: latency, launches and host work
        _layer("block_64x14_b1", "block", 1, 64, 14, 14, 64, 3, 1, 1),
        # AlexNet conv2 with the layers that follow it in the network (B-A-C-P with ReLU)
        _layer("alexnet_conv2_pool_b256", "block", 256, 96, 27, 27, 256, 5, 1, 2, relu=True, pool=True,
               w_std=0.01),
        # AlexNet conv4 in a training step's forward direction: the filters change every step
        _layer("alexnet_conv4_weights_b256", "block", 256, 384, 13, 13, 384, 3, 1, 1, weights=True,
               w_std=0.01),
        # second convolution of a ResNet-18 block of the first stage: large planes, shortcut added
        _layer("resnet_64x56_residual_b256", "block", 256, 64, 56, 56, 64, 3, 1, 1, residual=True),
        # the stride-2 layer that opens a stage, at the batch of a server
        _layer("resnet_64x56_stride2_b64", "block", 64, 64, 56, 56, 128, 3, 2, 1),
        # the widest point of the efficiency study: 1024 channels, 7x7 filters
        _layer("sweep_c1024_k7_b64", "block", 64, 1024, 14, 14, 256, 7, 1, 3),
        # nothing a multiple of anything: odd batch, planes, channels and filters
        _layer("ragged_100x15x17_b37", "block", 37, 100, 15, 17, 77, 5, 1, 2, valid=True),
        # 2-bit activations on a ResNet-18 layer
        _layer("kbit2_128x28_b256", "kbit", 256, 128, 28, 28, 128, 3, 1, 1, kbits=2),
        # binary weights only (the more accurate of the paper's two networks)
        _layer("bwn_256x14_b256", "bwn", 256, 256, 14, 14, 256, 3, 1, 1),
        # the gradient of a layer's input in a training step
        _layer("bgrad_128x28_b128", "bgrad", 128, 128, 28, 28, 128, 3, 1, 1),
        # the network's binary layers, one image (serving latency) and a full batch
        {"name": "chain_resnet18_b1", "kind": "chain", "N": 1},
        {"name": "chain_resnet18_b256", "kind": "chain", "N": 256},
    ]


# ---- drawing --------------------------------------------------------------------------------
_MAX_MACS = 160e9                  # per case, the sweep point's
_MAX_VALUES = 110e6                # inputs + outputs, the large ResNet layer's


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    return n if rng.random() < 0.3 else max(16, n // 16 * 16)      # most networks' are round


def _draw_layer(rng, kind):
    c = _layer("", kind, _log_int(rng, 1, 256), _channels(rng, 16, 1024), rng.randint(7, 56), 0,
               _channels(rng, 32, 512), 3, 1, 1)
    c["W"] = c["H"] if rng.random() < 0.6 else rng.randint(7, 56)
    if kind == "block" or kind == "kbit":
        c["k"] = rng.choice([1, 3, 3, 3, 5, 7])
        c["stride"] = rng.choice([1, 1, 1, 2])
        c["pad"] = c["k"] // 2
    if kind == "block":
        c["relu"] = rng.random() < 0.3
        c["pool"] = c["relu"] and rng.random() < 0.5
        c["residual"] = not c["pool"] and rng.random() < 0.3
        c["valid"] = rng.random() < 0.2
        c["weights"] = rng.random() < 0.3
    elif kind == "kbit":
        c["kbits"] = rng.choice([2, 2, 3, 4])
        c["N"] = (c["N"] + 3) // 4 * 4                    # the bit planes stay 16-byte aligned
    else:
        # the Binary-Weight kernel keeps a pixel tile's channels in shared memory
        c["C"] = _channels(rng, 16, 256)
        c["Co"] = _channels(rng, 32, 256)
    return c


def draw(rng):
    kind = rng.choice(["block"] * 6 + ["kbit", "bwn", "bgrad", "chain"])
    if kind == "chain":
        return {"kind": "chain", "N": _log_int(rng, 1, 200)}
    while True:
        c = _draw_layer(rng, kind)
        Ho, Wo = _out_hw(c)
        planes = c["C"] * c["H"] * c["W"] + (2 if c.get("residual") else 1) * c["Co"] * Ho * Wo
        if _macs(c) * c.get("kbits", 1) <= _MAX_MACS and c["N"] * planes <= _MAX_VALUES:
            del c["name"]
            return c


# ---- sizes ----------------------------------------------------------------------------------
def _out_hw(c):
    return ((c["H"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1,
            (c["W"] + 2 * c["pad"] - c["k"]) // c["stride"] + 1)


def _macs(c):
    Ho, Wo = _out_hw(c)
    return c["N"] * Ho * Wo * c["Co"] * c["C"] * c["k"] ** 2


def _pool_out(n):
    return (n - 3) // 2 + 1                              # AlexNet's overlapping 3x3 stride-2 pooling


def work(case):
    """Inputs read once, outputs written once; two operations per multiply-accumulate."""
    if case["kind"] == "chain":
        shapes = wl.chain_shapes(case["N"])
        first, last = shapes[0], shapes[-1]
        ho, wo = wl.out_hw(last)
        proj = [s for s in shapes if s.C_in != s.C_out]
        bits = sum(s.C_out * s.C_in * s.k ** 2 for s in shapes)
        return {"bytes": 4 * case["N"] * (first.C_in * first.H * first.W + last.C_out * ho * wo) + bits / 8 +
                4 * sum(s.C_in * s.C_out for s in proj),
                "flops": 2 * (sum(wl.macs(s) for s in shapes) + sum(wl.macs(s._replace(k=1, pad=0)) for s in proj))}
    c = case
    Ho, Wo = _out_hw(c)
    x, y = c["N"] * c["C"] * c["H"] * c["W"], c["N"] * c["Co"] * Ho * Wo
    filters = c["Co"] * c["C"] * c["k"] ** 2
    values = x + y * (2 if c.get("residual") else 1)
    if c.get("pool"):
        values += c["N"] * c["Co"] * _pool_out(Ho) * _pool_out(Wo)
    values += filters if c.get("weights") or c["kind"] == "bgrad" else filters / 32
    return {"bytes": 4 * values, "flops": 2 * _macs(c) * c.get("kbits", 1)}


def tolerance(case):
    # Sign bits, level codes and integer sums are exact; A, K, alpha and the outputs are fp32 sums
    # and products.  A chain's signs follow from fp32 values, so its outputs are as close only
    # where those values are the same.
    return {"rel": 1e-5}


# ---- one pass -------------------------------------------------------------------------------
def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))

    def normal(*shape, std=1.0):
        t = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
        return t.mul_(std) if std != 1.0 else t

    if case["kind"] == "chain":
        net = ChainRunner(case["N"])
        net.x0.copy_(normal(*net.x0.shape))
        for L in net.layers:
            L["w"].copy_(normal(*L["w"].shape, std=0.05))
        for P in net.proj.values():
            P["w"].copy_(normal(*P["w"].shape, std=0.05))
        net.binarize_weights()
        net.calibrate()                                  # BatchNorm statistics
        return {"case": case, "net": net}

    c = case
    d = X.make_desc(c["N"], c["C"], c["H"], c["W"], c["Co"], c["k"], c["k"], c["stride"], c["pad"],
                    (X.XNOR_FLAG_RELU if c.get("relu") else 0) |
                    (X.XNOR_FLAG_K_VALID_TAPS if c.get("valid") else 0))
    Ho, Wo = _out_hw(c)
    s = {"case": c, "d": d, "w": normal(c["Co"], c["C"], c["k"], c["k"], std=c["w_std"])}
    s["wp"], s["alpha"] = X.alloc_weights(c["Co"], c["C"], c["k"], c["k"])
    if c["kind"] == "bgrad":
        s["wT"] = X.alloc_weights_transposed(c["Co"], c["C"], c["k"], c["k"])
        s["gmax"], s["stream"], s["grad_in"] = X.alloc_bgrad(d)
        s["grad"] = normal(c["N"], c["Co"], Ho, Wo, std=0.01)
        return s
    X.xnor_binarize_weights(s["w"], s["wp"], s["alpha"])
    s["x"] = normal(c["N"], c["C"], c["H"], c["W"])
    s["scale"] = normal(c["C"], std=0.1).add_(1.0)
    s["shift"] = normal(c["C"], std=0.1)
    s["res"] = normal(c["N"], c["Co"], Ho, Wo) if c.get("residual") else None
    s["out"] = X.alloc_out(d)
    xp, s["A"], s["K"] = X.alloc_binactiv(d)
    if c["kind"] == "bwn":
        s["stream"] = X.alloc_bwn_input(d)
    elif c["kind"] == "kbit":
        s["x"].mul_(0.6)                                 # most values inside [-1, 1]
        s["xp"] = torch.empty((c["kbits"],) + tuple(xp.shape), dtype=torch.int32, device="cuda")
    else:
        s["xp"] = xp
    if c.get("pool"):
        s["pooled"] = torch.empty((c["N"], c["Co"], _pool_out(Ho), _pool_out(Wo)), device="cuda")
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "chain":
        return s["net"].forward()
    d, wp, alpha, K = s["d"], s["wp"], s["alpha"], s.get("K")
    if c["kind"] == "bgrad":
        X.xnor_binarize_weights(s["w"], wp, alpha)
        X.xnor_binarize_weights_transposed(s["w"], s["wT"])
        X.xnor_binary_gradient_backward(s["grad"], s["wT"], alpha, d, s["gmax"], s["stream"], s["grad_in"])
        return s["grad_in"], s["gmax"]
    if c["kind"] == "bwn":
        X.xnor_bwn_prepare_input(s["x"], s["scale"], s["shift"], d, s["stream"])
        X.xnor_bwn_conv2d_forward(s["stream"], wp, alpha, s["res"], d, s["out"])
        return s["out"]
    if c["kind"] == "kbit":
        X.xnor_binactiv_kbit(s["x"], s["scale"], s["shift"], d, c["kbits"], s["xp"], s["A"], K)
        X.xnor_conv2d_forward_kbit(s["xp"], c["kbits"], wp, alpha, K, s["res"], d, s["out"])
        return s["out"]
    if c.get("weights"):
        X.xnor_binarize_weights(s["w"], wp, alpha)
    X.xnor_binactiv(s["x"], s["scale"], s["shift"], d, s["xp"], s["A"], K)
    X.xnor_conv2d_forward(s["xp"], wp, alpha, K, s["res"], d, s["out"])
    if c.get("pool"):
        X.xnor_maxpool2d(s["out"], 3, 2, 0, False, s["pooled"])
        return s["pooled"]
    return [s["out"], wp, alpha] if c.get("weights") else s["out"]
