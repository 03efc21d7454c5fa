"""The work that programs built on this library have it do, as cases that can be timed and compared.

Five kinds of work, all through the public entry points (``LPNetwork`` and the functions of
``binding``), all on synthetic tensors with the distributions of the workloads: He-normal weights,
N(0, 0.01) biases, normal or uniform images, ReLU'd normal activations (about half zeros).

  net      one forward pass of a stack whose decimal points are fixed (paper Sec. 2.1), or its
           calibration; the stacks are the ones of ``workloads``
  conv     one LPConvolution call, alone or with the 2x2 max-pool after it
  ip       one LPInnerProduct call
  act      the quantizer / LPAct on an fp32 tensor or on a stored one, deterministic or stochastic
  measure  the range measurement and the bit-occupancy histogram of an fp32 tensor

Everything the library computes is an integer that is fixed bit for bit, so outputs compare exactly.
"""
import math

import torch

from paper_1711_04713_b200 import binding as B
from paper_1711_04713_b200 import workloads as wl
from paper_1711_04713_b200.network import LPNetwork, act_c_stride

STACKS = {          # specs, input height = width, input channels
    "lenet": (wl.lenet_specs, 28, 1),
    "giga1net": (wl.giga1net_specs, 224, 3),
    "vgg16": (wl.vgg16_specs, 224, 3),
}
MAX_BATCH = {"lenet": 2048, "giga1net": 256, "vgg16": 64}     # of drawn cases; twice that at 8 bits and fewer


def _net(name, stack, batch, n_bits, requantize=True, stochastic=False, calibrate=False):
    return {"name": name, "kind": "net", "stack": stack, "batch": batch, "n_bits": n_bits, "requantize": requantize,
            "stochastic": stochastic, "calibrate": calibrate}


def listed():
    return [
        # The small digit network on a handful of images: ten short launches, all latency.
        _net("lenet_n16_b8", "lenet", 8, 16),
        # One image through the large network with the parameters kept quantized: the latency of serving.
        _net("vgg16_n16_b1_serving", "vgg16", 1, 16, requantize=False),
        # The headline workload: a full batch, parameters quantized anew in every forward pass (Sec. 2.1).
        _net("vgg16_n16_b64", "vgg16", 64, 16),
        # The same stack at 8 bits, parameters kept: the throughput of serving.
        _net("vgg16_n8_b128_serving", "vgg16", 128, 8, requantize=False),
        # The paper's own network with stochastic rounding in every layer (Sec. 2.4), an ordinary batch.
        _net("giga1net_n16_b16_stochastic", "giga1net", 16, 16, stochastic=True),
        # Fixing every decimal point on a batch (Sec. 2.1, 2.3): a range pass and a storing pass per layer.
        _net("vgg16_n16_b16_calibrate", "vgg16", 16, 16, calibrate=True),
        # One layer of a network of the user's own: odd image sizes, channels that fill no whole tile.
        {"name": "conv3x3_ragged_n12", "kind": "conv", "N": 12, "H": 45, "W": 37, "C": 96, "K": 168, "R": 3, "pad": 1,
         "stride": 1, "nx": 12, "nw": 12, "pool": False},
        # The first inner product of the precision sweep, a large batch at 8 bits.
        {"name": "ip_25088_4096_n8_b256", "kind": "ip", "M": 256, "Kin": 25088, "K": 4096, "nx": 8, "nw": 8},
        # A classifier head on a few rows, output count no multiple of anything.
        {"name": "ip_4096_1000_n16_b5", "kind": "ip", "M": 5, "Kin": 4096, "K": 1000, "nx": 16, "nw": 16},
        # LPAct on a large fp32 activation (64 x 56 x 56 pixels of 256 channels) with ReLU and counters.
        {"name": "act_f32_relu_n16", "kind": "act", "outer": 200704, "inner": 256, "source": "f32", "n_bits": 16, "relu": True,
         "stochastic": False},
        # Stochastic quantization of a tensor whose channels need padding (50 -> 64).
        {"name": "act_f32_stochastic_padded_n16", "kind": "act", "outer": 150001, "inner": 50, "source": "f32", "n_bits": 16,
         "relu": False, "stochastic": True},
        # The statistics behind a thresholded allocation, over a weight tensor of odd size.
        {"name": "measure_7000003", "kind": "measure", "numel": 7000003, "n_bits": 16},
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["net", "net", "net", "conv", "conv", "ip", "ip", "act", "act", "measure"])
    width = lambda: rng.choice([4, 6, 8, 8, 10, 12, 14, 16, 16, 16])  # noqa: E731
    if kind == "net":
        stack, n = rng.choice(sorted(STACKS)), width()
        how = rng.choice(["forward", "forward", "serving", "serving", "stochastic", "calibrate"])
        most = MAX_BATCH[stack] * (2 if n <= 8 else 1)
        if how in ("stochastic", "calibrate"):
            most //= 2          # these passes do about twice the work per image
        c = _net("", stack, _log(rng, 1, most), n, how == "forward" or how == "stochastic", how == "stochastic",
                 how == "calibrate")
        del c["name"]
        return c
    if kind == "conv":
        while True:
            c = {"kind": "conv", "N": _log(rng, 1, 64), "H": _log(rng, 7, 224), "W": _log(rng, 7, 224), "C": _log(rng, 3, 512),
                 "K": _log(rng, 8, 512), "R": rng.choice([1, 3, 3, 3, 5]), "stride": rng.choice([1, 1, 1, 2]),
                 "nx": width(), "nw": 0, "pool": rng.random() < 0.25}
            c["pad"] = rng.choice([0, c["R"] // 2, c["R"] // 2])
            c["nw"] = c["nx"] if rng.random() < 0.8 else width()
            if c["pool"]:       # 2x2 windows need an even output
                c["stride"] = 1
                c["H"] += (c["H"] + 2 * c["pad"] - c["R"] + 1) % 2
                c["W"] += (c["W"] + 2 * c["pad"] - c["R"] + 1) % 2
            w = work(c)
            if w["flops"] <= 4e11 and w["bytes"] <= 1e9:
                return c
    if kind == "ip":
        n = width()
        c = {"kind": "ip", "M": _log(rng, 1, 512), "Kin": _log(rng, 64, 25088), "K": _log(rng, 10, 4096), "nx": n}
        c["nw"] = n if rng.random() < 0.8 else width()
        return c
    if kind == "act":
        inner = rng.choice([rng.randint(1, 64), 16 * rng.randint(1, 32), 512])
        return {"kind": "act", "outer": max(1, _log(rng, 1 << 12, 1 << 26) // inner), "inner": inner,
                "source": rng.choice(["f32", "f32", "q"]), "n_bits": width(), "relu": rng.random() < 0.5,
                "stochastic": rng.random() < 0.35}
    return {"kind": "measure", "numel": _log(rng, 1 << 10, 1 << 26), "n_bits": width()}


# --------------------------------------------------------------------------- preparation
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(shape, std, g):
    return torch.empty(shape, device="cuda").normal_(0.0, std, generator=g)


def _stack_params(specs, g):
    out = []
    for sp in specs:
        if sp.type == "pool":
            out.append({"type": "pool", "name": sp.name})
            continue
        shape = (sp.cout, sp.ksize, sp.ksize, sp.cin) if sp.type == "conv" else (sp.cout, sp.cin)
        fan_in = sp.cin * (sp.ksize * sp.ksize if sp.type == "conv" else 1)
        p = {"type": sp.type, "name": sp.name, "w": _normal(shape, math.sqrt(2.0 / fan_in), g).cpu().numpy(),
             "b": _normal((sp.cout,), 0.01, g).cpu().numpy(), "relu": sp.relu}
        if sp.type == "conv":
            p.update(pad=sp.pad, stride=sp.stride)
        out.append(p)
    return out


def _quantized(x, outer, inner, n_bits, pitch, with_q16=False):
    """A tensor stored with the decimal point of its own range."""
    mx = torch.zeros(1, device="cuda")
    fmt = torch.zeros(2, dtype=torch.int32, device="cuda")
    B.adaption_measure_range(x, n_bits, mx, fmt)
    q = B.QTensor.empty(outer, inner, n_bits, int(fmt.cpu()[1]), pitch, with_q16)
    B.adaption_quantize(x, outer, inner, q)
    return q


def _prepare_layer(case, seed):
    g = _gen(seed)
    nx, nw = case["nx"], case["nw"]
    if case["kind"] == "conv":
        N, H, W, C, K, R = (case[k] for k in ("N", "H", "W", "C", "K", "R"))
        pitch = act_c_stride(C)
        x = _quantized(_normal((N * H * W, C), 1.0, g).clamp_(min=0), N * H * W, C, nx, pitch)
        w = _quantized(_normal((K * R * R, C), math.sqrt(2.0 / (R * R * C)), g), K * R * R, C, nw, pitch)
        shape = B.conv_shape(N, H, W, C, K, R, R, case["pad"], case["stride"])
        oh, ow = _out_hw(case)
        rows, out_pitch = N * oh * ow, act_c_stride(K)
        need = B.adaption_lp_conv_workspace_bytes(shape, x.fmt(), w.fmt(), pitch)
    else:
        M, Kin, K = case["M"], case["Kin"], case["K"]
        x = _quantized(_normal((M, Kin), 1.0, g).clamp_(min=0), M, Kin, nx, None)
        w = _quantized(_normal((K, Kin), math.sqrt(2.0 / Kin), g), K, Kin, nw, None)
        shape, rows, out_pitch = None, M, B.pad_to(K, 16)
        need = B.adaption_lp_ip_workspace_bytes(M, Kin, K, x.fmt(), w.fmt())
    b = B.QTensor.empty(1, K, nw, w.frac_bits, None, True)
    B.adaption_quantize(_normal((K,), 0.01, g), 1, K, b)
    stats = B.new_stats()
    ws = torch.empty(need, dtype=torch.uint8, device="cuda") if need else None
    s = {"case": case, "shape": shape, "x": x, "w": w, "b": b, "stats": stats, "ws": ws, "y": None}
    # the output's decimal point: measured on this very layer (Sec. 2.3)
    _layer_call(s, B.MODE_RANGE)
    f = B.adaption_choose_frac_bits_from_acc(int(B.read_stats(stats).max_abs_acc), x.frac_bits + w.frac_bits, nx)
    if case.get("pool"):
        y = B.QTensor.empty(rows // 4, K, nx, f, out_pitch)
        need = B.adaption_lp_conv_pool_workspace_bytes(shape, x.fmt(), w.fmt(), y.fmt(), x.c_stride, out_pitch)
        s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    else:
        y = B.QTensor.empty(rows, K, nx, f, out_pitch)
    s["y"] = y
    stats.zero_()
    return s


def _layer_call(s, mode):
    c = s["case"]
    if c["kind"] == "ip":
        B.adaption_lp_ip_fwd(c["M"], c["Kin"], c["K"], s["x"], s["w"], s["b"].q16, s["b"].frac_bits, True, mode, B.ALGO_AUTO,
                             s["y"], s["stats"], s["ws"])
    elif c["pool"] and mode == B.MODE_REQUANT:
        B.adaption_lp_conv_pool_fwd(s["shape"], s["x"], s["w"], s["b"].q16, s["b"].frac_bits, True, B.ALGO_AUTO, s["y"],
                                    s["stats"], s["ws"])
    else:
        B.adaption_lp_conv_fwd(s["shape"], s["x"], s["w"], s["b"].q16, s["b"].frac_bits, True, mode, B.ALGO_AUTO, s["y"],
                               s["stats"], s["ws"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("conv", "ip"):
        return _prepare_layer(case, seed)
    g = _gen(seed)
    if kind == "net":
        specs, hw, channels = STACKS[case["stack"]]
        net = LPNetwork(_stack_params(specs(), g), case["batch"], (hw, hw), channels, case["n_bits"],
                        rounding_seed=seed if case["stochastic"] else None)
        x = torch.empty((case["batch"] * hw * hw, channels), device="cuda")
        x = x.uniform_(generator=g) if case["stack"] == "lenet" else x.normal_(generator=g)
        if not case["calibrate"]:
            net.calibrate(x)
            net.zero_stats()
        return {"case": case, "net": net, "x": x}
    if kind == "act":
        outer, inner, n = case["outer"], case["inner"], case["n_bits"]
        x, q = _normal((outer, inner), 1.0, g), None
        if case["source"] == "q":
            x, q = None, _quantized(x, outer, inner, n, None)
        f = max(0, n - 4) if q is None else max(0, q.frac_bits - 2)
        return {"case": case, "x": x, "q": q, "y": B.QTensor.empty(outer, inner, n, f), "stats": B.new_stats(), "seed": seed}
    return {"case": case, "x": _normal((case["numel"],), 0.7, g), "max": torch.zeros(1, device="cuda"),
            "fmt": torch.zeros(2, dtype=torch.int32, device="cuda"), "hist": B.new_hist()}


# --------------------------------------------------------------------------- one pass
def _planes(q):
    return [q.lo] if q.hi is None else [q.lo, q.hi]


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "net":
        net = state["net"]
        if c["calibrate"]:
            rec = net.calibrate(state["x"])
            formats = [r["frac_bits"] for r in rec]
            ranges = [r.get("max_abs_acc", 0) for r in rec]
            return {"formats": torch.tensor(formats), "ranges": torch.tensor(ranges), "logits": _planes(net.layers[-1].y),
                    "counters": [L.stats for L in net.layers if L.stats is not None]}
        y, _ = net.forward(state["x"], requantize_params=c["requantize"])
        # logits, and the counters of the sparsity report (they accumulate over the batches)
        return {"logits": _planes(y), "counters": [net.x_stats] + [L.stats for L in net.layers if L.stats is not None],
                "input_range": net.x_max_dev}
    if kind in ("conv", "ip"):
        _layer_call(state, B.MODE_REQUANT)
        return {"y": _planes(state["y"]), "counters": state["stats"]}
    if kind == "act":
        y, st, x, q = state["y"], state["stats"], state["x"], state["q"]
        if c["stochastic"]:
            B.adaption_lp_act_stochastic(x, q, c["outer"], c["inner"], c["relu"], y, state["seed"], None, st)
        else:
            B.adaption_lp_act(x, q, c["outer"], c["inner"], c["relu"], y, None, B.ROUND_DETERMINISTIC, st)
        return {"y": _planes(y), "counters": st}
    state["max"].zero_()
    state["hist"].zero_()
    B.adaption_measure_range(state["x"], c["n_bits"], state["max"], state["fmt"])
    B.adaption_bit_histogram(state["x"], state["hist"])
    return {"max": state["max"], "fmt": state["fmt"], "hist": state["hist"]}


# --------------------------------------------------------------------------- work and tolerance
def _out_hw(c):
    return tuple((c[d] + 2 * c["pad"] - c["R"]) // c["stride"] + 1 for d in ("H", "W"))


def _plane_bytes(n_bits):
    return 2 if n_bits > 8 else 1


def work(case):
    """Bytes: each operand read once, each result written once.  Operations: one multiply and one add per
    product of the layer, whatever the width (a 16-bit product is four 8-bit ones on the hardware)."""
    kind = case["kind"]
    if kind == "net":
        specs, hw, ch = STACKS[case["stack"]]
        p, b = _plane_bytes(case["n_bits"]), case["batch"]
        macs = params = 0
        h, last = hw, 0
        for sp in specs():
            if sp.type == "pool":
                h //= 2
            elif sp.type == "conv":
                h = (h + 2 * sp.pad - sp.ksize) // sp.stride + 1
                n = sp.cout * sp.ksize * sp.ksize * sp.cin
                macs, params = macs + n * h * h * b, params + n + sp.cout
            else:
                macs, params, last = macs + sp.cin * sp.cout * b, params + sp.cin * sp.cout + sp.cout, sp.cout
        per_param = 4 + p if case["requantize"] or case["calibrate"] else p
        # (calibrating runs every layer once to measure and once to store)
        return {"bytes": params * per_param + b * hw * hw * ch * 4 + b * last * p,
                "flops": 2.0 * macs * (2 if case["calibrate"] else 1)}
    if kind == "conv":
        oh, ow = _out_hw(case)
        m, k = case["N"] * oh * ow, case["R"] * case["R"] * case["C"]
        out = m * case["K"] // (4 if case["pool"] else 1)
        px, pw = _plane_bytes(case["nx"]), _plane_bytes(case["nw"])
        return {"bytes": case["N"] * case["H"] * case["W"] * case["C"] * px + case["K"] * k * pw + out * px,
                "flops": 2.0 * m * k * case["K"]}
    if kind == "ip":
        px, pw = _plane_bytes(case["nx"]), _plane_bytes(case["nw"])
        return {"bytes": case["M"] * case["Kin"] * px + case["K"] * case["Kin"] * pw + case["M"] * case["K"] * px,
                "flops": 2.0 * case["M"] * case["Kin"] * case["K"]}
    if kind == "act":
        p = _plane_bytes(case["n_bits"])
        return {"bytes": case["outer"] * case["inner"] * ((4 if case["source"] == "f32" else p) + p), "flops": 0}
    return {"bytes": case["numel"] * 4, "flops": 0}


def tolerance(case):
    return "exact"
