"""The workloads that this library's speed is judged on.

A case is a dict of plain values; its "kind" says which work it is:

  ternarize  fp32 master weights -> packed codes, scale and counts: per layer, per filter (Algorithm 1
             as printed) or binary (the BPWN baseline); what a training step does first and a
             deployment does once.
  update     the SGD step on the master weights and the coding sweep of the next iteration.
  gemm       a fully connected layer on codes that were packed once: inference.
  conv       a convolution layer on codes that were packed once: inference.
  layer      everything that a training step does for one convolution layer: codes, their re-layout,
             forward, backward through the ReLU and the affine, backward for data, weight gradient.
  net        a whole network of `nets`: a forward pass, or a training step, called directly or as the
             captured CUDA graph that a training loop of fixed shape replays.

Sizes are those of the networks in `nets`, of the GEMM sweep and of the ternarization benchmark in
bench.py, with their neighbours: odd batches, widths that are not multiples of a tile, single images.
"""
from __future__ import annotations

import math

import torch

from paper_1605_04711_b200 import nets, twn

DELTA = 0.7
SGD = {"lr": 0.01, "momentum": 0.9, "weight_decay": 1e-4}


def listed():
    return [
        # the second convolution of LeNet-5: the smallest call of a training step
        {"name": "ternarize_lenet_conv2", "kind": "ternarize", "rule": "layer", "rows": 64, "cols": 800},
        # 1e8 weights in one tensor: the size the ternarization bandwidth is quoted at
        {"name": "ternarize_1e8", "kind": "ternarize", "rule": "layer", "rows": 12288, "cols": 8192},
        # a fourth-stage 3x3 layer of the 1.5x wider ResNet-18, one threshold per filter
        {"name": "ternarize_filters_768x6912", "kind": "ternarize", "rule": "filter", "rows": 768, "cols": 6912},
        # the first fully connected layer of VGG-7 between two training iterations
        {"name": "update_vgg_fc1", "kind": "update", "rows": 1024, "cols": 8192},
        # the first fully connected layer of LeNet-5 for one image: a served request
        {"name": "gemm_1x1024x512", "kind": "gemm", "M": 1, "K": 1024, "N": 512, "code": 2, "out": "f32"},
        # a deep reduction with few outputs, and an odd row count (the sweep's 4096 x 4608 x 512 has its neighbours)
        {"name": "gemm_4001x4608x512", "kind": "gemm", "M": 4001, "K": 4608, "N": 512, "code": 2, "out": "f32"},
        # the largest shape of the GEMM sweep
        {"name": "gemm_16384x4096x4096", "kind": "gemm", "M": 16384, "K": 4096, "N": 4096, "code": 2, "out": "bf16"},
        # a third-stage 3x3 layer of ResNet-18 on binary weights, a request of a few images
        {"name": "conv_b1_14x14x256_b8", "kind": "conv", "B": 8, "H": 14, "Cin": 256, "Cout": 256, "k": 3, "stride": 1, "code": 1},
        # a strided layer of the wider ResNet-18 while it is trained, with a batch that fills no tile evenly
        {"name": "layer_28x28x192_384_s2_b50", "kind": "layer", "B": 50, "H": 28, "Cin": 192, "Cout": 384, "k": 3, "stride": 2},
        # LeNet-5 on a test batch: a few kernels of microseconds each
        {"name": "lenet5_forward_b100", "kind": "net", "net": "lenet5", "batch": 100, "train": False, "graph": False},
        # VGG-7 on a test batch
        {"name": "vgg7_forward_b128", "kind": "net", "net": "vgg7", "batch": 128, "train": False, "graph": False},
        # the training step of ResNet-18 at the paper's batch per GPU
        {"name": "resnet18_train_b64", "kind": "net", "net": "resnet18", "batch": 64, "train": True, "graph": True},
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(multiple, int(round(v / multiple)) * multiple)


def draw(rng):
    kind = rng.choice(["ternarize", "update", "gemm", "gemm", "conv", "conv", "layer", "layer", "net", "net"])
    if kind == "ternarize":
        rule = rng.choice(["layer", "layer", "filter", "binary"])
        rows = _log_int(rng, 10, 12288)
        return {"kind": kind, "rule": rule, "rows": rows, "cols": _log_int(rng, 25, min(24576, 100_000_000 // rows))}
    if kind == "update":
        rows = _log_int(rng, 10, 4096)
        return {"kind": kind, "rows": rows, "cols": _log_int(rng, 25, min(9216, 30_000_000 // rows))}
    if kind == "gemm":
        K, N = _log_int(rng, 64, 8192), _log_int(rng, 10, 4096, rng.choice([1, 8, 64]))
        return {"kind": kind, "M": _log_int(rng, 1, min(16384, 2 ** 38 // (K * N)), rng.choice([1, 1, 16])), "K": K, "N": N,
                "code": rng.choice([2, 2, 2, 1]), "out": rng.choice(["f32", "bf16", "bf16"])}
    if kind in ("conv", "layer"):
        code = 2 if kind == "layer" else rng.choice([2, 2, 1])
        k = rng.choice([1, 3, 3, 3, 5])
        stride = rng.choice([1, 1, 2])
        cin, cout = _log_int(rng, 32, 768, 32), _log_int(rng, 32, 768, 16)
        most = 6e10 if kind == "conv" else 2.5e10      # multiply-adds of one pass over the layer
        H = _log_int(rng, max(k, 7), 112)
        per_image = ((H + stride - 1) // stride) ** 2 * k * k * cin * cout
        while per_image > most:
            H = max(7, H // 2)
            per_image = ((H + stride - 1) // stride) ** 2 * k * k * cin * cout
        return {"kind": kind, "B": _log_int(rng, 1, max(1, min(128, int(most / per_image)))), "H": H, "Cin": cin, "Cout": cout,
                "k": k, "stride": stride, **({"code": code} if kind == "conv" else {})}
    net = rng.choice(["lenet5", "vgg7", "resnet18", "resnet18"])
    train = net == "resnet18" and rng.random() < 0.7
    return {"kind": kind, "net": net, "batch": _log_int(rng, 1, {"lenet5": 256, "vgg7": 160, "resnet18": 48}[net]),
            "train": train, "graph": rng.random() < 0.5}


# ---------------------------------------------------------------------- what a user has in hand
def _normal(g, *shape, std=1.0):
    return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(0.0, std, generator=g)


def _activations(g, *shape):
    """Outputs of a ReLU: half of them zero."""
    return _normal(g, *shape).relu_().to(torch.bfloat16)


def _gradients(g, *shape):
    return _normal(g, *shape, std=0.01).to(torch.bfloat16)


def _affine(g, n):
    return _normal(g, n, std=0.3).add_(1.0), _normal(g, n, std=0.3)


def _bytes(n):
    return torch.empty((max(int(n), 16) + 255) // 256 * 256, dtype=torch.uint8, device="cuda")


def _codes(g, rows, cols, bits, weights=None):
    """He-normal master weights and everything their ternarization (or binarization) writes."""
    s = {"rows": rows, "cols": cols, "W": _normal(g, rows, cols, std=math.sqrt(2.0 / cols)) if weights is None else weights}
    s["ld"] = twn.ld_for(cols) if bits == 2 else twn.ld_for_b1(cols)
    s["packed"] = torch.zeros((rows, s["ld"] * bits // 32), dtype=torch.int32, device="cuda")
    s["stats"] = twn.new_stats()
    s["ws"] = _bytes(max(twn.ternarize_workspace_bytes(), twn.binarize_workspace_bytes()))
    return s


def _stats_out(stats):
    """A twn_stats_t as its numbers: four doubles, then the counts and the status."""
    return {"sums": stats[..., :4].view(torch.float64), "counts": stats[..., 4:]}


def _encode(s, bits):
    if bits == 2:
        twn.ternarize(s["W"], DELTA, s["stats"], s["packed"], s["ld"], None, s["ws"])
    else:
        twn.binarize(s["W"], s["stats"], s["packed"], s["ld"], s["ws"])


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return {"case": case, **globals()["_prepare_" + case["kind"]](case, g, seed)}


def _prepare_ternarize(c, g, seed):
    s = _codes(g, c["rows"], c["cols"], 1 if c["rule"] == "binary" else 2)
    if c["rule"] == "filter":
        s["stats"] = twn.new_stats_rows(c["rows"])
    s["out"] = {"packed": s["packed"], **_stats_out(s["stats"])}
    return s


def _prepare_update(c, g, seed):
    s = _codes(g, c["rows"], c["cols"], 2)
    s["dW"] = _normal(g, c["rows"], c["cols"], std=1e-3)
    s["V"] = _normal(g, c["rows"], c["cols"], std=1e-3)
    s["out"] = {"W": s["W"], "V": s["V"], "packed": s["packed"], **_stats_out(s["stats"])}
    return s


def _prepare_gemm(c, g, seed):
    s = _codes(g, c["N"], c["K"], c["code"])
    _encode(s, c["code"])
    s["ldx"] = (c["K"] + 7) // 8 * 8
    s["X"] = torch.zeros((c["M"], s["ldx"]), dtype=torch.bfloat16, device="cuda")
    s["X"][:, :c["K"]] = _activations(g, c["M"], c["K"])
    s["scale"], s["shift"] = _affine(g, c["N"])
    f32 = c["out"] == "f32"
    s["Y"] = torch.zeros((c["M"], c["N"]), dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    # logits come as fp32 with no ReLU, hidden layers as bf16 after the folded batch norm and a ReLU
    s["epi"] = (twn.epilogue(out_dtype=twn.F32) if f32 else
                twn.epilogue(s["scale"], s["shift"], relu=True, out_dtype=twn.BF16))
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


def _prepare_conv(c, g, seed):
    K = c["k"] * c["k"] * c["Cin"]
    bits = c.get("code", 2)
    s = _codes(g, c["Cout"], K, bits)
    s["desc"] = d = twn.conv_desc(c["B"], c["H"], c["H"], c["Cin"], c["Cout"], c["k"], c["stride"], c["k"] // 2)
    s["X"] = _activations(g, c["B"], c["H"], c["H"], c["Cin"])
    s["Y"] = torch.zeros((c["B"], d.Ho, d.Wo, c["Cout"]), dtype=torch.bfloat16, device="cuda")
    s["scale"], s["shift"] = _affine(g, c["Cout"])
    s["epi"] = twn.epilogue(s["scale"], s["shift"], relu=True, out_dtype=twn.BF16)
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    _encode(s, bits)
    return s


def _prepare_layer(c, g, seed):
    s = _prepare_conv(c, g, seed)
    d = s["desc"]
    s["dY"] = _gradients(g, c["B"], d.Ho, d.Wo, c["Cout"])
    s["dZ"] = torch.zeros_like(s["dY"])
    s["dX"] = torch.zeros_like(s["X"])
    s["dW"] = torch.zeros((c["Cout"], s["cols"]), dtype=torch.float32, device="cuda")
    s["ld_b"] = twn.ld_for(c["k"] * c["k"] * c["Cout"])
    s["packed_b"] = torch.zeros((c["Cin"], s["ld_b"] // 16), dtype=torch.int32, device="cuda")
    s["epi_b"] = twn.epilogue(out_dtype=twn.BF16)
    s["ws_dw"] = _bytes(twn.conv2d_bwd_weight_workspace_bytes(d))
    s["out"] = {"Y": s["Y"], "dX": s["dX"], "dW": s["dW"], "packed": s["packed"], **_stats_out(s["stats"])}
    return s


def _prepare_net(c, g, seed):
    make = getattr(nets, c["net"])
    net = make(batch=c["batch"], train=c["train"], seed=seed)
    net.act["input"].copy_(_normal(g, *net.act["input"].shape))
    s = {"net": net}
    last = net.ops[-1][1]
    s["out"] = [net.act[last.name]]
    if c["train"]:
        s["dlogits"] = _gradients(g, c["batch"], last.Cout)
        s["out"] += [L.extra["dW"] for L in net.layers.values()]
        step = lambda: net.train_step(s["dlogits"])     # noqa: E731
    else:
        net.ternarize_all()
        step = net.forward
    s["step"] = step
    if c["graph"]:
        step()
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"], stream=torch.cuda.Stream(priority=-1)):
            step()
        s["step"] = s["graph"].replay
    return s


# ---------------------------------------------------------------------- one pass
def run(s):
    return globals()["_run_" + s["case"]["kind"]](s)


def _run_ternarize(s):
    rule = s["case"]["rule"]
    if rule == "layer":
        twn.ternarize(s["W"], DELTA, s["stats"], s["packed"], s["ld"], None, s["ws"])
    elif rule == "filter":
        twn.ternarize_rows(s["W"], DELTA, s["stats"], s["packed"], s["ld"])
    else:
        twn.binarize(s["W"], s["stats"], s["packed"], s["ld"], s["ws"])
    return s["out"]


def _run_update(s):
    twn.sgd_update(s["W"], s["dW"], s["V"], SGD["lr"], SGD["momentum"], SGD["weight_decay"], DELTA, s["stats"], s["ws"])
    twn.ternarize_codes(s["W"], s["rows"], s["cols"], s["stats"], s["packed"], s["ld"], None, s["ws"])
    return s["out"]


def _run_gemm(s):
    c = s["case"]
    call = twn.gemm if c["code"] == 2 else twn.gemm_b1
    call(s["X"], s["ldx"], s["packed"], s["ld"], s["stats"], c["M"], c["N"], c["K"], s["epi"], s["Y"], c["N"], s["status"])
    return s["Y"]


def _run_conv(s):
    call = twn.conv2d_fwd if s["case"]["code"] == 2 else twn.conv2d_fwd_b1
    call(s["desc"], s["X"], s["packed"], s["ld"], s["stats"], s["epi"], s["Y"], s["status"])
    return s["Y"]


def _run_layer(s):
    d, status = s["desc"], s["status"]
    twn.ternarize(s["W"], DELTA, s["stats"], s["packed"], s["ld"], None, s["ws"])
    twn.transpose_codes(s["packed"], s["ld"], d, s["packed_b"], s["ld_b"])
    twn.conv2d_fwd(d, s["X"], s["packed"], s["ld"], s["stats"], s["epi"], s["Y"], status)
    twn.act_bwd(s["dY"], s["Y"], s["scale"], s["dY"].numel(), d.Cout, s["dZ"])
    twn.conv2d_bwd_data(d, s["dZ"], s["packed_b"], s["ld_b"], s["stats"], s["epi_b"], s["dX"], status)
    twn.conv2d_bwd_weight(d, s["X"], s["dZ"], s["dW"], s["ws_dw"], status)
    return s["out"]


def _run_net(s):
    s["step"]()
    return s["out"]


# ---------------------------------------------------------------------- what a pass cannot do without
_NET_OPS = {"lenet5": nets.lenet5_ops, "vgg7": nets.vgg7_ops, "resnet18": nets.resnet18_ops}


def work(case):
    c, kind = case, case["kind"]
    if kind == "ternarize":
        n = c["rows"] * c["cols"]
        code = 0.125 if c["rule"] == "binary" else 0.25
        return {"bytes": n * (4 + code) + (64 * c["rows"] if c["rule"] == "filter" else 64), "flops": 0}
    if kind == "update":
        return {"bytes": c["rows"] * c["cols"] * 20.25 + 64, "flops": 0}
    if kind == "gemm":
        out = 4 if c["out"] == "f32" else 2
        return {"bytes": 2 * c["M"] * c["K"] + c["N"] * c["K"] * c["code"] / 8 + out * c["M"] * c["N"],
                "flops": 2 * c["M"] * c["N"] * c["K"]}
    if kind in ("conv", "layer"):
        d = twn.conv_desc(c["B"], c["H"], c["H"], c["Cin"], c["Cout"], c["k"], c["stride"], c["k"] // 2)
        x, y = c["B"] * c["H"] ** 2 * c["Cin"], c["B"] * d.Ho * d.Wo * c["Cout"]
        n = c["k"] ** 2 * c["Cin"] * c["Cout"]
        flops = 2 * y * c["k"] ** 2 * c["Cin"]
        if kind == "conv":
            return {"bytes": 2 * (x + y) + n * c["code"] / 8, "flops": flops}
        # W, X, dY in; codes, Y, dX, dW out
        return {"bytes": n * (4 + 0.25 + 4) + 2 * (x + y) + 2 * (y + x), "flops": 3 * flops}
    # weights (or their codes), images and the gradient of the logits in; logits and weight gradients out
    layers = [op[1] for op in _NET_OPS[c["net"]]() if op[0] == "layer"]
    for L in layers:
        L.B, L.K = c["batch"], L.k * L.k * L.Cin
    first, last = layers[0], layers[-1]
    n = sum(L.K * L.Cout for L in layers)
    macs = sum(L.macs for L in layers)
    io = c["batch"] * (2 * first.H * first.W * first.Cin + 4 * last.Cout)
    if not c["train"]:
        return {"bytes": n / 4 + io, "flops": 2 * macs}
    return {"bytes": 8.25 * n + io + 2 * c["batch"] * last.Cout, "flops": 2 * (3 * macs - first.macs)}


def tolerance(case):
    kind = case["kind"]
    if kind in ("ternarize", "update"):
        return {"rel": 1e-12}           # codes and counts are exact, the sums are fp64
    if kind == "gemm" and case["out"] == "f32":
        return {"rel": 1e-5}            # exact products, fp32 accumulation
    if kind == "net" and case["train"]:
        return {"rel": 2e-2}            # bf16 activations and gradients through twenty layers and their ReLU gates
    return {"rel": 1e-2}                # bf16 results
