"""Performance cases of the quantized-convolution library: what its users have it do, through its public entry points.

Five kinds of work:

  layer      one int8 layer, `QConv.run` on a handle that is kept
  fp_layer   one layer on 8-bit floating-point operands, `QConvNP.run` on a handle that is kept
  network    int8 inference of a calibrated network: `QNetwork.run` (captured, or part of a batch without a graph) or
             `QNetwork.run_pipelined` (batches in pinned host memory, results back to it)
  calibrate  the offline procedure on a whole network, `QNetwork.calibrate`
  tensor     one tensor's statistics, threshold search, conversion and (floating-point types) the conversion back

`listed()` names twelve such cases, `draw(rng)` makes more of the same ranges.  Inputs are synthetic and made from the
seed alone; shapes are those of the networks in `workloads.py`, or generic.
"""
import math

import numpy as np
import torch

from paper_1805_07941_b200 import binding, workloads
from paper_1805_07941_b200.network import QNetwork

_OUT_MODES = {"int8": binding.OUT_INT8, "int32": binding.OUT_INT32, "float": binding.OUT_FLOAT}
_FAMILIES = {"resnet50": workloads.resnet50, "vgg16": workloads.vgg16, "inception": workloads.inception,
             "mobilenet": workloads.mobilenet}
# The largest batch of each network: the repository's benchmark sizes.
_MAX_BATCH = {"resnet50": 32, "vgg16": 64, "inception": 128, "mobilenet": 256}
_NBINS = 2048


def _layer(name, N, H, W, C, K, R=3, stride=1, depthwise=False, residual=False, relu=True, rounding=0, out="int8",
           per_channel=True, n_run=None):
    case = dict(kind="layer", N=N, n_run=N if n_run is None else n_run, H=H, W=W, C=C, K=K, R=R, stride=stride,
                depthwise=depthwise, residual=residual, relu=relu, rounding=rounding, out=out, per_channel=per_channel)
    return dict(case, name=name) if name else case


def _fp_layer(name, N, H, W, C, K, R=3, stride=1, p=4, relu=True):
    case = dict(kind="fp_layer", N=N, H=H, W=W, C=C, K=K, R=R, stride=stride, p=p, relu=relu)
    return dict(case, name=name) if name else case


def _network(name, family, batch, res, how="graph", n_run=None, batches=1):
    case = dict(kind="network", family=family, batch=batch, res=res, how=how, n_run=batch if n_run is None else n_run,
                batches=batches)
    return dict(case, name=name) if name else case


def _calibrate(name, family, batch, res, images, threshold=None):
    case = dict(kind="calibrate", family=family, batch=batch, res=res, images=images, threshold=threshold or "max")
    return dict(case, name=name) if name else case


def _tensor(name, count, p=4, measure="l1", relu=True):
    case = dict(kind="tensor", count=count, p=p, measure=measure, relu=relu)
    return dict(case, name=name) if name else case


def listed():
    return [
        # The one-layer configuration: the smallest call there is, where launch and host path are all of the time.
        _layer("conv_tiny", 1, 32, 32, 16, 16, per_channel=False),
        # Odd image, odd batch, channels no tile divides, a residual and the rounding mode that is not the default.
        _layer("conv_ragged", 13, 35, 27, 96, 200, residual=True, rounding=1),
        # A mid-size 3x3 layer on the 8-bit floating-point type with 4 significand bits, which the paper recommends.
        _fp_layer("conv_fp8", 32, 28, 28, 128, 128),
        # Inference of one image: a request at a time, latency and launches count.
        _network("resnet50_one", "resnet50", 1, 224),
        # The four networks at the batch they are benchmarked at: throughput.
        _network("resnet50", "resnet50", 32, 224),
        _network("vgg16", "vgg16", 64, 224),
        _network("inception", "inception", 128, 28),
        _network("mobilenet", "mobilenet", 256, 224),
        # The last, shorter batch of a data set: fewer images than the graph was recorded for.
        _network("resnet50_tail", "resnet50", 32, 224, how="partial", n_run=21),
        # End to end: batches arrive in pinned host memory and results go back to it.
        _network("resnet50_host", "resnet50", 32, 224, how="host", batches=4),
        # Deployment: float weights and one batch of images in, every exponent and the int8 layers out.
        _calibrate("calibrate_resnet50", "resnet50", 32, 224, 32),
        # One activation tensor (ResNet-50 stage-1 output, batch 32): statistics, Algorithm 1, codes and back.
        _tensor("tensor_fp8", 32 * 56 * 56 * 256),
    ]


# ---------------------------------------------------------------------------------------------------- drawing
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_layer(rng):
    while True:
        R = rng.choice([1, 1, 3, 3, 3, 5])
        H, W = _log(rng, 7, 112), _log(rng, 7, 112)
        C = 16 * _log(rng, 1, 64)
        depthwise = R == 3 and rng.random() < 0.2
        K = C if depthwise else rng.choice([16 * _log(rng, 1, 64), _log(rng, 10, 1000)])
        N = _log(rng, 1, 64)
        stride = rng.choice([1, 1, 1, 2])
        plain = depthwise or rng.random() < 0.6
        out = "int8" if plain else rng.choice(["int8", "int8", "int32", "float"])
        case = _layer(None, N, H, W, C, K, R=R, stride=stride, depthwise=depthwise,
                      residual=not depthwise and rng.random() < 0.3, relu=rng.random() < 0.7,
                      rounding=0 if plain else rng.choice([0, 1, 2, 3]), out=out, per_channel=rng.random() < 0.5,
                      n_run=N if rng.random() < 0.8 else max(1, N - 1))
        w = work(case)
        if w["flops"] < 5e11 and w["bytes"] < 5e8:
            return case


def _draw_fp_layer(rng):
    while True:
        case = _fp_layer(None, _log(rng, 1, 64), _log(rng, 7, 56), _log(rng, 7, 56), 16 * _log(rng, 1, 32),
                         rng.choice([16 * _log(rng, 1, 32), _log(rng, 10, 500)]), R=rng.choice([1, 3, 3]),
                         stride=rng.choice([1, 1, 2]), p=rng.choice([4, 4, 3]), relu=rng.random() < 0.7)
        w = work(case)
        if w["flops"] < 1e11 and w["bytes"] < 2e8:
            return case


def _draw_network(rng):
    family = rng.choice(sorted(_FAMILIES))
    batch = _log(rng, 1, _MAX_BATCH[family])
    res = rng.randint(14, 28) if family == "inception" else 16 * rng.randint(6, 14)
    how = rng.choice(["graph", "graph", "graph", "partial", "host"])
    if how == "partial":
        batch = max(2, batch)
        return _network(None, family, batch, res, how=how, n_run=rng.randint(1, batch - 1))
    return _network(None, family, batch, res, how=how, batches=4 if how == "host" else 1)


def _draw_calibrate(rng):
    family = rng.choice(["resnet50", "inception", "mobilenet"])
    images = _log(rng, 4, 32)
    res = rng.randint(14, 28) if family == "inception" else 32 * rng.randint(3, 7)
    return _calibrate(None, family, images, res, images, threshold=rng.choice([None, None, "l1"]))


def _draw_tensor(rng):
    return _tensor(None, _log(rng, 1000, 1e8), p=rng.choice([3, 4, 7]), measure=rng.choice(["l1", "ks", "cvm", "kl"]),
                   relu=rng.random() < 0.6)


def draw(rng):
    return rng.choice([_draw_layer] * 4 + [_draw_network] * 4 + [_draw_fp_layer] * 2 + [_draw_tensor] * 2 +
                      [_draw_calibrate])(rng)


# ---------------------------------------------------------------------------------------------------- preparing
def _out_hw(case):
    pad = case["R"] // 2
    return (workloads.out_size(case["H"], case["R"], case["stride"], pad),
            workloads.out_size(case["W"], case["R"], case["stride"], pad))


def _activations(gen, shape, relu=True):
    """int8 codes as a calibrated layer leaves them: (half-)normal, the largest near the end of the range."""
    x = torch.randn(shape, generator=gen, device="cuda") * 32.0
    return (x.abs() if relu else x).round_().clamp_(-127, 127).to(torch.int8)


def _prepare_layer(case, gen):
    P, Q = _out_hw(case)
    N, C, K, R = case["N"], case["C"], case["K"], case["R"]
    cg = 1 if case["depthwise"] else C
    w = _activations(gen, (K, R, R, cg), relu=False).cpu().numpy()
    bias = torch.randint(-2**12, 2**12, (K,), generator=gen, device="cuda").cpu().numpy().astype(np.int32)
    # the shift that takes three standard deviations of the sum to the end of the output's range
    base = max(1, round(math.log2(3.0 * 32.0 * 32.0 * math.sqrt(R * R * cg) / 127.0)))
    spread = torch.randint(-1, 2, (K,), generator=gen, device="cuda").cpu().numpy()
    shift = np.clip(base + (spread if case["per_channel"] else 0 * spread), 0, 31).astype(np.int32)
    res = _activations(gen, (N, P, Q, K)) if case["residual"] else None
    lshift = np.clip(shift - 1, 0, 23).astype(np.int32) if case["residual"] else None
    mode = _OUT_MODES[case["out"]]
    conv = binding.QConv(w, bias, shift, lshift, np.full(K, -12, np.int32) if case["out"] == "float" else None,
                         N=N, H=case["H"], W=case["W"], C=C, K=K, R=R, S=R, stride_h=case["stride"],
                         stride_w=case["stride"], pad_h=R // 2, pad_w=R // 2, groups=C if case["depthwise"] else 1,
                         relu=int(case["relu"]), rounding=case["rounding"], out_mode=mode,
                         has_residual=int(case["residual"]))
    y = torch.empty((case["n_run"], P, Q, K), device="cuda",
                    dtype={"int8": torch.int8, "int32": torch.int32, "float": torch.float32}[case["out"]])
    x = _activations(gen, (N, case["H"], case["W"], C))
    return dict(kind="layer", conv=conv, x=x[:case["n_run"]], y=y, res=None if res is None else res[:case["n_run"]])


def _fp_codes(gen, shape, e, p):
    return binding.qquantize_f32_np(torch.randn(shape, generator=gen, device="cuda"), e, 8, p)


def _prepare_fp_layer(case, gen):
    P, Q = _out_hw(case)
    N, C, K, R, p = case["N"], case["C"], case["K"], case["R"], case["p"]
    # five standard deviations at the end of the range of the operand types
    e = math.ceil(math.log2(5.0 / _beta_max(8, p)))
    w = _fp_codes(gen, (K, R, R, C), e, p).cpu().numpy()
    bias = torch.randint(-2**16, 2**16, (K,), generator=gen, device="cuda").cpu().numpy().astype(np.int32)
    sums = math.sqrt(R * R * C) * (_beta_max(8, p) / 5.0) ** 2
    shift = np.full(K, max(0, round(math.log2(5.0 * sums / _beta_max(8, p)))), np.int32)
    conv = binding.QConvNP(w, bias, shift, N=N, H=case["H"], W=case["W"], C=C, K=K, R=R, S=R, stride_h=case["stride"],
                           stride_w=case["stride"], pad_h=R // 2, pad_w=R // 2, n_in=8, p_in=p, n_w=8, p_w=p, n_out=8,
                           p_out=p, relu=int(case["relu"]))
    return dict(kind="fp_layer", conv=conv, x=_fp_codes(gen, (N, case["H"], case["W"], C), e, p),
                y=torch.empty((N, P, Q, K), dtype=torch.uint8, device="cuda"))


def _net(case):
    return _FAMILIES[case["family"]](batch=case["batch"], res=case["res"])


def _float_weights(net, gen):
    """The float model: normal weights at the deviation workloads.py gives each layer, zero where channels are padding."""
    weights = {}
    for nd in net["nodes"]:
        if nd["op"] != "conv":
            continue
        cg = nd["C"] // nd["groups"]
        w = torch.randn((nd["K"], nd["R"], nd["S"], cg), generator=gen, device="cuda") * nd["w_std"]
        if nd["groups"] == 1:
            w[..., nd["C_real"]:] = 0
        b = torch.randn((nd["K"],), generator=gen, device="cuda") * nd["b_std"]
        weights[nd["name"]] = (w.cpu().numpy(), b.cpu().numpy())
    return weights


def _images(net, gen, n):
    x = torch.randn((n,) + tuple(net["input"][1:]), generator=gen, device="cuda")
    return x.abs_() if net["input_dist"] == "halfnormal" else x


def _prepare_network(case, gen):
    net = _net(case)
    qn = QNetwork(net, _float_weights(net, gen))
    x = _images(net, gen, case["n_run"])
    qn.calibrate(x[:min(8, case["n_run"])])
    qn.capture()
    state = dict(kind="network", how=case["how"], net=qn)
    if case["how"] == "host":
        hosts = [x.cpu().pin_memory()]
        hosts += [_images(net, gen, case["batch"]).cpu().pin_memory() for _ in range(case["batches"] - 1)]
        shape = qn.bufs[qn.last].shape
        outs = [torch.empty(shape, dtype=torch.int8).pin_memory() for _ in range(case["batches"])]
        return dict(state, hosts=hosts, outs=outs)
    return dict(state, x=x)


def _prepare_calibrate(case, gen):
    net = _net(case)
    qn = QNetwork(net, _float_weights(net, gen))
    threshold = None if case["threshold"] == "max" else case["threshold"]
    return dict(kind="calibrate", net=qn, x=_images(net, gen, case["images"]), threshold=threshold)


def _beta_max(n, p):
    """Largest value of the n-bit type with p significand bits."""
    return 2**(n - 1) - 1 if p == n - 1 else ((2 << p) - 1) * 2**((1 << (n - p - 1)) - 2)


def _prepare_tensor(case, gen):
    x = torch.randn((case["count"],), generator=gen, device="cuda")
    return dict(kind="tensor", x=x.relu_() if case["relu"] else x, p=case["p"], measure=case["measure"],
                scale=127.0 / _beta_max(8, case["p"]))


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return {"layer": _prepare_layer, "fp_layer": _prepare_fp_layer, "network": _prepare_network,
            "calibrate": _prepare_calibrate, "tensor": _prepare_tensor}[case["kind"]](case, gen)


# ---------------------------------------------------------------------------------------------------- running
def _run_calibrate(state):
    qn = state["net"].calibrate(state["x"], threshold=state["threshold"])
    small = [np.array([qn.e_buf[k] for k in sorted(qn.e_buf)], np.int32)]
    weights = []
    for name in sorted(qn.params):
        par = qn.params[name]
        weights.append(par["wq"])
        small += [par[k] for k in ("e_w", "bias_q", "acc_exp", "shift", "res_lshift") if par[k] is not None]
    return dict(exponents=np.concatenate(small), weights=weights, activations=qn.bufs[qn.last][:state["x"].shape[0]])


def _run_tensor(state):
    x, p = state["x"], state["p"]
    st = binding.qcalib_collect(x, _NBINS)
    gamma, delta = binding.qthreshold_search(st["hist"], st["maxabs"], 8, p, state["measure"])
    e = binding.qscale_exponent(gamma * state["scale"])
    out = dict(maxabs=st["maxabs"], count=st["count"], nonfinite=st["nonfinite"], sum=st["sum"], sumsq=st["sumsq"],
               hist=st["hist"].view(np.int64), gamma=gamma, delta=delta)
    if p == 7:
        return dict(out, codes=binding.qquantize_f32(x, e))
    codes = binding.qquantize_f32_np(x, e, 8, p)
    return dict(out, codes=codes, values=binding.qdequantize_np(codes, e, 8, p))


def run(state):
    kind = state["kind"]
    if kind == "layer":
        return state["conv"].run(state["x"], state["y"], state["res"])
    if kind == "fp_layer":
        return state["conv"].run(state["x"], state["y"])
    if kind == "calibrate":
        return _run_calibrate(state)
    if kind == "tensor":
        return _run_tensor(state)
    if state["how"] == "host":
        state["net"].run_pipelined(state["hosts"], state["outs"])
        return state["outs"]
    return state["net"].run(state["x"])


# ---------------------------------------------------------------------------------------------------- accounting
def work(case):
    """Bytes and operations of one pass.  A layer: its tensors and weights once.  A network: every layer's, since it runs
    layer by layer and its activations are larger than the caches at the batches it is used at, and the float image."""
    kind = case["kind"]
    if kind == "tensor":
        # read once for the statistics and the codes; codes written; codes read and values written on the way back
        back = 0 if case["p"] == 7 else 5
        return dict(bytes=(5 + back) * case["count"] + 8 * _NBINS, flops=4 * case["count"])
    if kind in ("layer", "fp_layer"):
        P, Q = _out_hw(case)
        n = case.get("n_run", case["N"])
        cg = 1 if case.get("depthwise") else case["C"]
        weights = case["K"] * case["R"] * case["R"] * cg
        outs = n * P * Q * case["K"]
        size = {"int8": 1, "int32": 4, "float": 4}[case.get("out", "int8")]
        moved = n * case["H"] * case["W"] * case["C"] + weights + 4 * case["K"] + outs * size
        return dict(bytes=moved + (outs if case.get("residual") else 0), flops=2 * outs * case["R"] * case["R"] * cg)
    net = _net(case)
    n = case["images"] if kind == "calibrate" else case["n_run"]
    convs = [nd for nd in net["nodes"] if nd["op"] == "conv"]
    moved = sum(workloads.conv_alg_bytes(nd, n) for nd in convs)
    ops = 2 * sum(workloads.conv_macs(nd, n) for nd in convs)
    moved += 4 * n * int(np.prod(net["input"][1:]))
    if kind == "calibrate":
        # the float weights are read, and every layer runs twice: once in floats for its statistics (written and read)
        moved += sum(4 * nd["K"] * nd["R"] * nd["S"] * nd["C"] // nd["groups"] for nd in convs)
        moved += sum(workloads.conv_alg_bytes(nd, n) + 7 * n * nd["P"] * nd["Q"] * nd["K"] for nd in convs)
        ops *= 2
    return dict(bytes=moved * case.get("batches", 1), flops=ops * case.get("batches", 1))


def tolerance(case):
    """Everything is integers and exact, but a tensor's sums and the search's measure, which are float64 sums whose order
    is the implementation's own; float outputs of a layer are exact functions of an integer."""
    if case["kind"] == "tensor":
        return {"rel": 1e-9, "max": 1e-9}
    return "exact"
