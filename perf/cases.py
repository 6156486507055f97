"""Performance cases of the integer training framework.

Every case is one call sequence that a program makes through the public
binding: a training step of a chain of local-loss blocks, a forward of such a
chain, one kernel-level contraction layer, an integer matrix product, the
pre-processing of a dataset, and the allocation-free conv forward.  All results
are integers, so every case is compared exactly.

A network is written as text: blocks separated by ``|``, layers by spaces,
``c64`` a 3x3 conv to 64 channels, ``c64p`` the same followed by the 2x2
max-pool, ``l100`` a linear layer to 100 features; the output block follows.

Weights are uniform in [-w, w] (``w`` for the first layer of a block, ``w_deep``
for the layers after it, ``w_lr`` for the learning and output layers).  About 10
is a network just initialised; after some hundred steps single-layer blocks
hold some hundreds, and blocks of two convs millions in the first (its gradient
comes through the second) and some ten thousands in the second.  The inverse learning
rate ``gamma`` is 512, times 3 for every plateau passed; the later one keeps the
weights in that range over the many passes of a measurement.  Images are normal
with sigma 64, clamped to [-127, 127], as the integer pre-processing leaves
them; labels are uniform.
"""
import math

import numpy as np
import torch

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import workloads as wl

ALPHA_INV = 10
M64 = (1 << 64) - 1


# ------------------------------------------------------------------ the cases
def net_text(name):
    """The network of one of the repository's workloads, as text."""
    blocks = []
    for b in wl.WORKLOADS[name]["blocks"]:
        if b["layers"]:
            blocks.append(" ".join(("c%d%s" % (l[2], "p" if l[5] else "")) if l[0] == wl.CONV
                                   else "l%d" % l[2] for l in b["layers"]))
    return "|".join(blocks)


def train(name, net, hw, chans, batch, w, w_lr, w_deep=None, classes=10, graph=False, fused=False,
          trunc=False, d_lr=0, eta_fw=0, eta_lr=0, dropout=0, gamma=512):
    return {"name": name, "kind": "train", "net": net, "hw": hw, "chans": chans, "batch": batch,
            "w": w, "w_deep": w if w_deep is None else w_deep, "w_lr": w_lr, "classes": classes,
            "graph": graph, "fused": fused, "trunc": trunc, "d_lr": d_lr, "eta_fw": eta_fw, "eta_lr": eta_lr, "dropout": dropout,
            "gamma": gamma}


def listed():
    return [
        # the smallest network in use, a digit classifier's MLP at the paper's batch: launches and latency
        train("train_mlp_small", net_text("mlp_784_100_50_10_b64"), 28, 1, 64, 600, 60),
        # a small CNN on 28 x 28 images, one channel in, 14 x 14 maps that no tile divides
        train("train_cnn_small", net_text("cnn_32_64_b64"), 28, 1, 64, 600, 60, trunc=True,
              gamma=512 * 27),
        # the paper's wide MLP with its weight decay and dropout: linear layers, 3000 features
        train("train_mlp_wide", net_text("mlp4_cifar10_b64"), 32, 1, 64, 600, 60, eta_fw=19000,
              eta_lr=7500, dropout=6554, gamma=512 * 27),
        # the paper's smaller VGG at its batch and hyper-parameters: an ordinary training step
        train("train_vgg8b", net_text("vgg8b_cifar10_b64"), 32, 3, 64, 600, 60, d_lr=4096,
              eta_fw=25000, eta_lr=3000, dropout=9830, trunc=True, gamma=512 * 27),
        # the benchmark's network as its driver runs it: two convs a block, a
        # stream per block, one CUDA graph, deltas that fill 32 bits
        train("train_vgg_style_graph", net_text("vgg_64_128_256_b128"), 32, 3, 128, 5000000, 300,
              w_deep=10000, graph=True, trunc=True, gamma=512 * 729),
        # one block of a user's own shape: channels, maps and batch that no tile
        # divides, more classes than the fused learning kernels hold, truncated updates
        train("train_block_odd", "c48 c80p", 18, 40, 37, 600, 60, classes=47, trunc=True),
        # inference on one image: eager launches of a whole network, latency
        {"name": "forward_vgg8b_b1", "kind": "forward", "net": net_text("vgg8b_cifar10_b64"), "hw": 32,
         "chans": 3, "batch": 1, "w": 600, "w_deep": 600},
        # evaluation of a test set in large batches through the paper's larger VGG
        {"name": "forward_vgg11b_b256", "kind": "forward", "net": net_text("vgg11b_cifar10_b64"),
         "hw": 32, "chans": 3, "batch": 256, "w": 600, "w_deep": 600},
        # one layer's three contractions as kernels, at a size of the sweep
        {"name": "contract_b256_16_256", "kind": "contract", "h": 16, "w": 16, "cin": 256,
         "cout": 256, "batch": 256, "w_max": 30000, "d_max": 1 << 20},
        # the integer matrix product at a size of the sweep
        {"name": "gemm_4096", "kind": "gemm", "m": 4096, "n": 4096, "k": 4096, "w_max": 30000},
        # a colour image training set, raw bytes in, int8 out
        {"name": "prep_50000", "kind": "prep", "n": 50000 * 32 * 32 * 3, "values": "natural"},
        # one conv layer inside a program that may not allocate
        {"name": "noalloc_b8_16_64", "kind": "noalloc", "h": 16, "w": 16, "cin": 64, "cout": 64,
         "batch": 8, "pool": True, "w_max": 4000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["train_mlp", "train_conv", "train_conv", "forward", "forward", "contract",
                       "gemm", "prep", "noalloc"])
    w = rng.choice([10, 600, 600, 4000])
    if kind == "train_mlp":
        widths = [_log(rng, 48, 3000) for _ in range(rng.randint(1, 4))]
        if rng.random() < 0.6:
            widths = [8 * max(6, v // 8) for v in widths]
        return train("", "|".join("l%d" % v for v in widths), rng.randint(14, 40), 1,
                     _log(rng, 8, 256), w, 60, classes=rng.choice([2, 10, 10, 10, 26]), gamma=512 * 27,
                     fused=rng.random() < 0.25, eta_fw=rng.choice([0, 25000]),
                     dropout=rng.choice([0, 6554]))
    if kind in ("train_conv", "forward"):
        blocks, hw = [], rng.randint(8, 40)
        size, chans = hw, rng.choice([1, 3, 3, 32, 64])
        for _ in range(rng.randint(1, 4)):
            layers = []
            for _ in range(rng.randint(1, 2)):
                layers.append("c%d" % (16 * rng.randint(2, 16)))
            if size >= 16 and rng.random() < 0.7:
                layers[-1] += "p"
                size //= 2
            blocks.append(" ".join(layers))
        net = "|".join(blocks)
        if kind == "forward":
            return {"kind": kind, "net": net, "hw": hw, "chans": chans, "batch": _log(rng, 1, 256),
                    "w": w, "w_deep": w}
        return train("", net, hw, chans, _log(rng, 4, 160), w, 60,
                     classes=rng.choice([10, 10, 10, 47]), gamma=512 * 27, graph=rng.random() < 0.25,
                     fused=rng.random() < 0.2, trunc=rng.random() < 0.3,
                     d_lr=rng.choice([0, 4096]), eta_fw=rng.choice([0, 25000]))
    if kind == "contract":
        return {"kind": kind, "h": rng.randint(7, 34), "w": rng.randint(7, 34),
                "cin": 16 * rng.randint(2, 24), "cout": 16 * rng.randint(2, 24),
                "batch": _log(rng, 4, 256), "w_max": rng.choice([100, 30000, 1 << 22]),
                "d_max": rng.choice([30000, 1 << 20, (1 << 31) - 1])}
    if kind == "gemm":
        return {"kind": kind, "m": _log(rng, 64, 6000), "n": _log(rng, 64, 6000),
                "k": 8 * _log(rng, 8, 700), "w_max": rng.choice([100, 30000, 1 << 22])}
    if kind == "prep":
        return {"kind": kind, "n": _log(rng, 1000, 150000000),
                "values": rng.choice(["natural", "digits"])}
    h, wd = rng.randint(4, 28), rng.randint(4, 28)
    cin, cout = rng.choice([1, 3, 16, 32, 64]), 8 * rng.randint(2, 16)
    batch = min(_log(rng, 1, 64), (1 << 21) // (h * wd * cout))
    return {"kind": kind, "h": h, "w": wd, "cin": cin, "cout": cout, "batch": max(1, batch),
            "pool": rng.random() < 0.5, "w_max": rng.choice([100, 4000])}


def draw(rng):
    """One more case of the same kinds, no more work than the largest listed one."""
    most = max(work(c)["flops"] for c in listed())
    while True:
        case = _draw(rng)
        case.pop("name", None)
        if work(case)["flops"] <= (most if case["kind"] in ("forward", "gemm") else most / 4):
            return case


# ------------------------------------------------------------------ networks
def blocks_of(case):
    """[(layers, in_features)] in the binding's layer tuples, the output block last."""
    size, chans, feat = case["hw"], case["chans"], case["hw"] ** 2 * case["chans"]
    out = []
    for text in case["net"].split("|"):
        layers, first = [], feat
        for word in text.split():
            n, pool = int(word[1:].rstrip("p")), word.endswith("p")
            if word[0] == "c":
                layers.append((nb.NITRO_CONV3X3, chans, n, size, size, pool))
                size, chans = size // 2 if pool else size, n
                feat = size * size * n
            else:
                layers.append((nb.NITRO_LINEAR, feat, n, 1, 1, False))
                feat = n
        out.append((layers, first))
    out.append(([], feat))
    return out


def lr_window(layer, d_lr):
    """Learning-layer pool window (kh, kw) of a block that ends in `layer`."""
    kind, _, c, h, w, pool = layer
    h, w, kh, kw = h // 2 if pool else h, w // 2 if pool else w, 1, 1
    if kind != nb.NITRO_CONV3X3 or d_lr <= 0:
        return 1, 1
    while c * (h // kh) * (w // kw) > d_lr:
        if kh <= kw and 2 * kh <= h:
            kh *= 2
        elif 2 * kw <= w:
            kw *= 2
        elif 2 * kh <= h:
            kh *= 2
        else:
            break
    return kh, kw


def lr_features(layers, in_features, d_lr):
    if not layers:
        return in_features
    kind, _, c, h, w, pool = layers[-1]
    if kind != nb.NITRO_CONV3X3:
        return c
    kh, kw = lr_window(layers[-1], d_lr)
    return c * ((h // 2 if pool else h) // kh) * ((w // 2 if pool else w) // kw)


def fan_in(layer):
    return (9 if layer[0] == nb.NITRO_CONV3X3 else 1) * layer[1]


def net_data(case, seed):
    """Images, labels and every block's weights, from the seed alone."""
    rng = np.random.default_rng([seed, 1])
    b = case["batch"]
    x = np.clip(np.rint(rng.normal(0, 64, (b, case["hw"] ** 2 * case["chans"]))), -127, 127)
    data = {"x": x.astype(np.int8), "w": [], "wlr": []}
    for layers, feat in blocks_of(case):
        data["w"].append([])
        for j, l in enumerate(layers):
            w = case["w_deep"] if j else case["w"]
            data["w"][-1].append(rng.integers(-w, w + 1, l[2] * fan_in(l), dtype=np.int32))
        if case["kind"] == "train":
            wl_, g = case["w_lr"], case["classes"]
            n = g * lr_features(layers, feat, case["d_lr"])
            data["wlr"].append(rng.integers(-wl_, wl_ + 1, n, dtype=np.int32))
    if case["kind"] == "train":
        data["y"] = rng.integers(0, case["classes"], b, dtype=np.int32)
    return data


def gradient(block, which, layer=0):
    """A view of the block's own gradient memory that keeps the block alive:
    the memory goes with the block, and outputs outlive the state."""
    t = block.grad_device(which, layer)
    t.block = block
    return t


class Net:
    """A chain of blocks with its inputs and buffers on the GPU."""

    def __init__(self, case, seed):
        self.case = case
        b, spec, data = case["batch"], blocks_of(case), net_data(case, seed)
        training = case["kind"] == "train"
        hyper = {}
        if training:
            hyper = dict(num_classes=case["classes"], alpha_inv=ALPHA_INV, gamma_inv_lr=case["gamma"],
                         eta_inv_fw=case["eta_fw"], eta_inv_lr=case["eta_lr"],
                         sgd_round=nb.NITRO_ROUND_TRUNC if case["trunc"] else nb.NITRO_ROUND_FLOOR,
                         d_lr=case["d_lr"], dropout_p16=case["dropout"])
        else:
            spec = spec[:-1]
        self.blocks = [nb.Block(l, f, seed=seed + i, max_batch=b, **hyper)
                       for i, (l, f) in enumerate(spec)]
        self.data = data
        self.set_weights()
        self.x = torch.from_numpy(data["x"]).cuda()
        self.acts = [self.x]
        for g in self.blocks:
            self.acts.append(torch.empty((b, g.out_features), dtype=torch.int8, device="cuda")
                             if g.layers else self.acts[-1])
        self.graph = None
        if training:
            self.y = torch.from_numpy(data["y"]).cuda()
            self.loss = torch.zeros(len(self.blocks), dtype=torch.int64, device="cuda")
            self.dw = [gradient(g, nb.NITRO_T_DW, i) for g in self.blocks
                       for i in range(len(g.layers))]
            self.dwlr = [gradient(g, nb.NITRO_T_DWLR) for g in self.blocks]
            if case["graph"]:
                self.capture()
        self.data = None

    def set_weights(self):
        for i, g in enumerate(self.blocks):
            for j in range(len(g.layers)):
                g.set(nb.NITRO_T_W, j, self.data["w"][i][j])
            if self.data["wlr"]:
                g.set(nb.NITRO_T_WLR, 0, self.data["wlr"][i])

    def capture(self):
        """One CUDA graph of the step, a stream per block, after two eager steps
        that settle the kernel variants; the weights are then put back."""
        self.streams = [torch.cuda.Stream() for _ in self.blocks]
        self.done = [torch.cuda.Event() for _ in self.blocks]
        for _ in range(2):
            self.step_streams()
        torch.cuda.synchronize()
        self.set_weights()
        for g in self.blocks:
            g.set(nb.NITRO_T_STEP, 0, np.zeros(1, np.uint32))
            g.status(clear=True)
        self.x_new, self.x = self.x, self.x.clone()   # a graph reads its own input buffers
        self.y_new, self.y = self.y, self.y.clone()
        self.acts[0] = self.x
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.stream(side), torch.cuda.graph(self.graph, stream=side):
            self.step_streams()
        torch.cuda.current_stream().wait_stream(side)

    def forward(self):
        for i, g in enumerate(self.blocks):
            g.forward(self.acts[i], self.acts[i + 1] if g.layers else None)

    def step(self):
        self.forward()
        for i, g in enumerate(self.blocks):
            if self.case["fused"]:
                g.backward_update(self.acts[i], self.y, self.loss[i:i + 1])
            else:
                g.backward(self.acts[i], self.y, self.loss[i:i + 1])
                g.sgd()

    def step_streams(self):
        """Every block on its own stream: a block's backward and update overlap
        the blocks after it, which wait only for its forward."""
        main = torch.cuda.current_stream()
        for i, (g, s) in enumerate(zip(self.blocks, self.streams)):
            s.wait_stream(main)
            if i:
                s.wait_event(self.done[i - 1])
            g.forward(self.acts[i], self.acts[i + 1] if g.layers else None, stream=s)
            self.done[i].record(s)
            if self.case["fused"]:
                g.backward_update(self.acts[i], self.y, self.loss[i:i + 1], stream=s)
            else:
                g.backward(self.acts[i], self.y, self.loss[i:i + 1], stream=s)
                g.sgd(stream=s)
        for s in self.streams:
            main.wait_stream(s)

    def run(self):
        if self.case["kind"] == "forward":
            self.forward()
            return {"act": self.acts[1:]}
        if self.graph is not None:
            self.x.copy_(self.x_new)
            self.y.copy_(self.y_new)
            self.graph.replay()
        else:
            self.step()
        return {"act": self.acts[1:-1], "loss": self.loss, "dw": self.dw, "dwlr": self.dwlr}


# ------------------------------------------------------------------ the other entry points
def conv_data(case, seed):
    rng = np.random.default_rng([seed, 2])
    b, h, w, ci, co = case["batch"], case["h"], case["w"], case["cin"], case["cout"]
    a = np.clip(np.rint(rng.normal(0, 64, (b, h, w, ci))), -127, 127).astype(np.int8)
    m = case["w_max"]
    wt = rng.integers(-m, m + 1, (co, 3, 3, ci), dtype=np.int32)
    if case["kind"] == "noalloc":
        return a, wt
    m = case["d_max"]
    return a, wt, rng.integers(-m, m, (b, h, w, co), dtype=np.int32, endpoint=True)


class Contract:
    def __init__(self, case, seed):
        b, h, w, ci, co = case["batch"], case["h"], case["w"], case["cin"], case["cout"]
        self.conv = nb.Conv3x3(b, h, w, ci, co)
        self.a, self.w, self.d = (torch.from_numpy(t).cuda() for t in conv_data(case, seed))
        new = lambda *shape: torch.empty(shape, dtype=torch.int64, device="cuda")  # noqa: E731
        self.z, self.dw, self.g = new(b, h, w, co), new(co, 3, 3, ci), new(b, h, w, ci)

    def run(self):
        self.conv.contract(nb.NITRO_CONTRACT_FWD, self.a, self.w, self.z)
        self.conv.contract(nb.NITRO_CONTRACT_WGRAD, self.a, self.d, self.dw)
        self.conv.contract(nb.NITRO_CONTRACT_DGRAD, self.d, self.w, self.g)
        return {"z": self.z, "dw": self.dw, "g": self.g}


def gemm_data(case, seed):
    rng = np.random.default_rng([seed, 3])
    m = case["w_max"]
    return (rng.integers(-127, 128, (case["m"], case["k"]), dtype=np.int8),
            rng.integers(-m, m + 1, (case["n"], case["k"]), dtype=np.int32))


class Gemm:
    def __init__(self, case, seed):
        self.gemm = nb.IntGemm(case["m"], case["n"], case["k"])
        self.a, self.b = (torch.from_numpy(t).cuda() for t in gemm_data(case, seed))
        self.c = torch.empty((case["m"], case["n"]), dtype=torch.int64, device="cuda")

    def run(self):
        return self.gemm.run(self.a, self.b, self.c)


def prep_data(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["n"]
    if case["values"] == "natural":
        x = torch.empty(n, device="cuda").normal_(120, 64, generator=gen)
        return x.round_().clamp_(0, 255).to(torch.uint8)
    x = torch.randint(1, 256, (n,), generator=gen, dtype=torch.uint8, device="cuda")
    return x * (torch.rand(n, generator=gen, device="cuda") > 0.8)


class Prep:
    def __init__(self, case, seed):
        self.prep = nb.IntPrep()
        self.x = prep_data(case, seed)
        self.out = torch.empty(case["n"], dtype=torch.int8, device="cuda")

    def run(self):
        self.prep.fit(self.x)
        return self.prep.apply(self.x, self.out)


class Noalloc:
    def __init__(self, case, seed):
        self.case = case
        self.a, self.w = (torch.from_numpy(t).cuda() for t in conv_data(case, seed))
        b, h, w, co = case["batch"], case["h"], case["w"], case["cout"]
        pooled = (b, h // 2, w // 2, co) if case["pool"] else (b, h, w, co)
        self.out = torch.empty(pooled, dtype=torch.int8, device="cuda")
        self.region = torch.empty((b, h, w, co), dtype=torch.int8, device="cuda")
        self.argmax = torch.empty(pooled, dtype=torch.int8, device="cuda") if case["pool"] else None

    def run(self):
        c = self.case
        st = nb.nitro_conv3x3_forward_noalloc(
            self.a.data_ptr(), self.w.data_ptr(), c["batch"], c["h"], c["w"], c["cin"], c["cout"],
            c["pool"], ALPHA_INV, self.out.data_ptr(), self.region.data_ptr(),
            self.argmax.data_ptr() if c["pool"] else None, torch.cuda.current_stream().cuda_stream)
        if st != nb.NITRO_OK:
            raise nb.NitroError(st, "nitro_conv3x3_forward_noalloc")
        return [self.out, self.region] + ([self.argmax] if c["pool"] else [])


KINDS = {"train": Net, "forward": Net, "contract": Contract, "gemm": Gemm, "prep": Prep,
         "noalloc": Noalloc}


def prepare(case, seed):
    return KINDS[case["kind"]](case, seed)


def run(state):
    return state.run()


# ------------------------------------------------------------------ work and tolerance
def work(case):
    kind = case["kind"]
    if kind in ("train", "forward"):
        b, by, ops = case["batch"], 0, 0
        by += b * case["hw"] ** 2 * case["chans"] + 4 * b
        for layers, feat in blocks_of(case):
            for i, l in enumerate(layers):
                pre = l[2] * (l[3] * l[4] if l[0] == nb.NITRO_CONV3X3 else 1)
                n = l[2] * fan_in(l)
                macs = b * pre * fan_in(l)
                if kind == "train":     # forward, weight gradient, input gradient inside the block
                    ops += 2 * macs * (3 if i else 2)
                    by += 16 * n        # W read and written, dW written
                else:
                    ops += 2 * macs
                    by += 4 * n
            if layers:
                l = layers[-1]
                by += b * l[2] * ((l[3] // 2) * (l[4] // 2) if l[5] else l[3] * l[4])
            if kind == "train":
                d = lr_features(layers, feat, case["d_lr"])
                ops += 2 * b * d * case["classes"] * (3 if layers else 2)
                by += 16 * d * case["classes"]
        return {"bytes": by, "flops": ops}
    if kind == "prep":      # fit, then apply: the data is read, then the map of it written
        return {"bytes": 2 * case["n"], "flops": 2 * case["n"]}
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": m * k + 4 * n * k + 8 * m * n, "flops": 2 * m * n * k}
    p = case["batch"] * case["h"] * case["w"]
    ci, co = case["cin"], case["cout"]
    if kind == "contract":
        return {"bytes": p * (ci + 4 * co) + 36 * ci * co + 8 * (p * (ci + co) + 9 * ci * co),
                "flops": 3 * 2 * p * 9 * ci * co}
    return {"bytes": p * (ci + 2 * co) + 36 * ci * co, "flops": 2 * p * 9 * ci * co}


def tolerance(case):
    return "exact"      # whole numbers throughout


# ------------------------------------------------------------------ exact results, plain torch
def i32(t):
    """The low 32 bits of int64 values, signed (how 32-bit storage wraps)."""
    return ((t + (1 << 31)) & 0xffffffff) - (1 << 31)


def mm(a, b):
    """a @ b of integers modulo 2^64: 16-bit halves, whose float64 products are whole."""
    def halves(t):
        lo = ((t + 32768) & 65535) - 32768
        hi = (t - lo) >> 16
        return [(0, lo.double())] + ([(16, hi.double())] if bool(hi.any()) else [])
    out = 0
    ha, hb = halves(a), halves(b)
    for sa, fa in ha:
        for sb, fb in hb:
            out = out + ((fa @ fb).to(torch.int64) << (sa + sb))
    return out


def taps(t, flip=False):
    """[B,H,W,C] -> [B*H*W, 9*C], the 3x3 neighbourhood of every pixel."""
    b, h, w, c = t.shape
    p = torch.nn.functional.pad(t, (0, 0, 1, 1, 1, 1))
    s = range(8, -1, -1) if flip else range(9)
    return torch.cat([p[:, k // 3:k // 3 + h, k % 3:k % 3 + w] for k in s], 3).reshape(b * h * w, 9 * c)


def relu(z):
    """NITRO-ReLU values and pieces of scaled pre-activations."""
    a = ALPHA_INV
    mu = ((-127) // a + (-127) // (2 * a) + 63 + 127) // 4
    v = torch.where(z < 0, z.clamp(min=-127) // a, z.clamp(max=127)) - mu
    return v, torch.where(z < -127, 0, torch.where(z < 0, 1, torch.where(z <= 127, 2, 3)))


def relu_back(g, region):
    return torch.where(region == 1, g // ALPHA_INV, torch.where(region == 2, g, 0))


def pool(t, kh, kw):
    """First maximum of kh x kw windows of [B,H,W,C] and its position."""
    b, h, w, c = t.shape
    oh, ow, n = h // kh, w // kw, kh * kw
    t = t[:, :oh * kh, :ow * kw].reshape(b, oh, kh, ow, kw, c).permute(0, 1, 3, 2, 4, 5)
    order = torch.arange(n - 1, -1, -1, device=t.device).reshape(n, 1)
    key = (t.reshape(b, oh, ow, n, c) * n + order).amax(3)
    return key // n, n - 1 - key % n


def unpool(g, pos, shape, kh, kw):
    """Gradients of pool() back to the window positions that won."""
    b, h, w, c = shape
    oh, ow = h // kh, w // kw
    k = torch.arange(kh * kw, device=g.device).reshape(kh * kw, 1)
    t = torch.where(pos[:, :, :, None] == k, g[:, :, :, None], 0)
    t = t.reshape(b, oh, ow, kh, kw, c).permute(0, 1, 3, 2, 4, 5).reshape(b, oh * kh, ow * kw, c)
    out = g.new_zeros(shape)
    out[:, :oh * kh, :ow * kw] = t
    return out


def splitmix(seed, index):
    """Outputs `index` (int64 tensor, modulo 2^64) of SplitMix64, top 16 bits."""
    def signed(v):
        return v - (1 << 64) if v >> 63 else v

    def rsh(t, n):
        return (t >> n) & ((1 << (64 - n)) - 1)
    z = (index + 1) * signed(0x9E3779B97F4A7C15) + signed(seed & M64)
    z = (z ^ rsh(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ rsh(z, 27)) * signed(0x94D049BB133111EB)
    return rsh(z ^ rsh(z, 31), 48)


def layer_forward(x, w, layer, drop=None):
    """One forward layer on [B, ...] int64: output, its inputs as matrix, pieces, pool positions."""
    kind, cin, cout, h, wd, pooled = layer
    b = x.shape[0]
    cols = taps(x.reshape(b, h, wd, cin)) if kind == nb.NITRO_CONV3X3 else x.reshape(b, cin)
    v, region = relu((mm(cols, w.reshape(cout, -1).T) >> 8) // fan_in(layer))
    if drop is not None:
        gone = splitmix(drop[0], torch.arange(v.numel(), device=v.device) + drop[1]) < drop[2]
        v, region = v.masked_fill(gone.reshape(v.shape), 0), region.masked_fill(gone.reshape(v.shape), 4)
    v, region, pos = v.reshape(b, h, wd, cout), region.reshape(b, h, wd, cout), None
    if pooled:
        v, pos = pool(v, 2, 2)
    return v, cols, region, pos


def exact_net(case, seed):
    data = net_data(case, seed)
    dev = lambda t: torch.from_numpy(t).cuda().to(torch.int64)  # noqa: E731
    x = dev(data["x"])
    out = {"act": [], "loss": [], "dw": [], "dwlr": []}
    for i, (layers, feat) in enumerate(blocks_of(case)):
        kept = []
        for j, l in enumerate(layers):
            drop = None
            if case.get("dropout") and l[0] == nb.NITRO_LINEAR:
                base = (1 << 63) + (j << 31)      # step 0 of the mask stream
                drop = (seed + i, base - (1 << 64), case["dropout"])
            x, cols, region, pos = layer_forward(x, dev(data["w"][i][j]), l, drop)
            kept.append((cols, region, pos))
        if layers:
            out["act"].append(x.reshape(x.shape[0], -1).to(torch.int8))
        if case["kind"] == "train":
            exact_backward(case, data, i, layers, x, kept, out)
    if case["kind"] == "forward":
        return {"act": out["act"]}
    out["loss"] = torch.stack(out["loss"])
    return out


def exact_backward(case, data, i, layers, x, kept, out):
    g, b = case["classes"], case["batch"]
    dev = lambda t: torch.from_numpy(t).cuda().to(torch.int64)  # noqa: E731
    kh, kw = lr_window(layers[-1], case["d_lr"]) if layers else (1, 1)
    a, apos = pool(x, kh, kw) if kh * kw > 1 else (x, None)
    flat = a.reshape(b, -1)
    wlr = dev(data["wlr"][i]).reshape(g, -1)
    onehot = torch.nn.functional.one_hot(dev(data["y"]), g)
    gl = i32((mm(flat, wlr.T) >> 8) // wlr.shape[1] - 32 * onehot)
    out["loss"].append((gl * gl).sum() // 2)
    out["dwlr"].append(mm(gl.T, flat).reshape(-1))
    if not layers:
        return
    grad = i32(mm(gl, wlr)).reshape(a.shape)
    if apos is not None:
        grad = unpool(grad, apos, x.shape, kh, kw)
    grads = []
    for j in range(len(layers) - 1, -1, -1):
        kind, cin, cout, h, wd, pooled = layers[j]
        cols, region, pos = kept[j]
        grad = grad.reshape(b, h // 2, wd // 2, cout) if pooled else grad.reshape(b, h, wd, cout)
        if pooled:
            grad = unpool(grad, pos, region.shape, 2, 2)
        delta = relu_back(grad, region)
        grads.append(mm(delta.reshape(-1, cout).T, cols).reshape(-1))
        if j:
            w = dev(data["w"][i][j]).reshape(cout, -1, cin)
            dcols = taps(delta, flip=True) if kind == nb.NITRO_CONV3X3 else delta.reshape(b, cout)
            grad = i32(mm(dcols, w.permute(1, 0, 2).reshape(-1, cin)))
    out["dw"].extend(reversed(grads))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "forward"):
        return exact_net(case, seed)
    if kind == "prep":
        x = prep_data(case, seed).to(torch.int64)
        mu = int(x.sum()) // x.numel()
        x -= mu
        omega = int(x.abs().sum()) // x.numel()
        return (x * 51 // max(omega, 1)).clamp(-127, 127).to(torch.int8)
    if kind == "gemm":
        a, b = (torch.from_numpy(t).cuda().to(torch.int64) for t in gemm_data(case, seed))
        return mm(a, b.T)
    a, w, *d = (torch.from_numpy(t).cuda().to(torch.int64) for t in conv_data(case, seed))
    ci, co = case["cin"], case["cout"]
    if kind == "noalloc":
        layer = (nb.NITRO_CONV3X3, ci, co, case["h"], case["w"], case["pool"])
        v, _, region, pos = layer_forward(a, w, layer)
        return [t.to(torch.int8) for t in ([v, region] + ([pos] if case["pool"] else []))]
    z = mm(taps(a), w.reshape(co, -1).T).reshape(*a.shape[:3], co)
    dw = mm(d[0].reshape(-1, co).T, taps(a)).reshape(co, 3, 3, ci)
    g = mm(taps(d[0], flip=True), w.reshape(co, 9, ci).permute(1, 0, 2).reshape(-1, ci))
    return {"z": z, "dw": dw, "g": g.reshape(*a.shape[:3], ci)}
