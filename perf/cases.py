"""What a program that trains with this library has it do, as cases to be timed.

A case is one pass through the public entry points of ``paper_2112_05387_b200``: a layer-parallel
training step (one call, the three calls, or replayed from a recorded graph), the step together with the
distillation of the AuxNets, layer-serial training, or evaluation.  The networks are those of
``workloads/configs.py``; batch size, image size, number of classes and module split vary as a program
varies them (training batch, small batch, last ragged batch, reduced training resolution).

Keys of a case
    net        workload that gives architecture, split and loss
    dtype      "bf16" | "f32": storage type of the activations
    batch, height, width, classes
    modules    0: the workload's own split, else the number of modules of nearly equal block count
    mode       "step"         lp_layer_parallel_step
               "three_calls"  lp_auxnet_forward, lp_modules_fwd_bwd_all, lp_step
               "distill"      lp_layer_parallel_step followed by lp_auxnet_distill
               "serial"       lp_serial_fwd_bwd, lp_step
               "eval"         lp_forward_serial
    loss       "penalty" | "al"
    momentum   0.0, or the momentum of the SGD update (weight decay 5e-4 goes with it)
    recursive  AuxNets as independent stacks instead of the serial chain
    graph      the pass is recorded once and replayed, as bench.py and long training runs do
"""
import numpy as np
import torch

import paper_2112_05387_b200 as lp
from workloads import get_config, with_modules

_LR, _LR_PREACT = 0.02, 0.004   # rates at which thousands of passes over one random batch stay finite
_LR_LAMBDA = 0.1     # correction of the auxiliary variables
_LR_AUX = 1e-3       # AuxNet distillation


def _case(name, net, batch, height=32, width=None, classes=10, dtype="bf16", modules=0, mode="step", loss="penalty",
          momentum=0.0, recursive=False, graph=True):
    case = dict(net=net, dtype=dtype, batch=batch, height=height, width=width or height, classes=classes,
                modules=modules, mode=mode, loss=loss, momentum=momentum, recursive=recursive, graph=graph)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest call there is: the tiny network of the smoke test, launched call by call
        _case("tiny_f32", "tiny", 8, 8, dtype="f32", loss="al", graph=False),
        # fp32 training of a CIFAR-sized network (the reference precision a user checks bf16 runs against)
        _case("resnet56_f32", "resnet56", 32, dtype="f32"),
        # CIFAR-shaped training at the workloads' own batch, recorded and replayed
        _case("resnet56", "resnet56", 128),
        _case("resnet110_al", "resnet110", 128, classes=100, loss="al"),
        # small-batch training with momentum and weight decay, the three calls enqueued one by one
        _case("resnet56_three_calls", "resnet56", 20, mode="three_calls", momentum=0.9, graph=False),
        # the whole of Algorithm 1, AuxNet distillation included, on an epoch's last ragged batch
        _case("resnet110_distill", "resnet110", 50, classes=100, loss="al", mode="distill"),
        # wide network: the benchmark's workload, and the layer-serial training it is compared with
        _case("wrn28_10", "wrn28_10", 128),
        _case("wrn28_10_serial", "wrn28_10", 64, mode="serial", graph=False),
        # ImageNet-shaped training at the workloads' own batches
        _case("resnet34_al", "resnet34", 64, 224, classes=1000, loss="al"),
        _case("resnet50", "resnet50", 32, 224, classes=1000),
        # evaluation of the last batch of a validation set, images that are not square
        _case("resnet34_eval", "resnet34", 37, 192, 256, classes=1000, mode="eval", graph=False),
        # reduced training resolution (176: the last stage works on 11x11 -> 6x6), recursive AuxNets
        _case("resnet50_176", "resnet50", 12, 176, classes=1000, recursive=True),
    ]


def draw(rng):
    """One more case of the same ranges."""
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    while True:
        net = rng.choice(["tiny", "resnet56", "resnet56", "resnet110", "resnet110", "wrn28_10", "wrn28_10",
                          "resnet34", "resnet34", "resnet50", "resnet50"])
        if net == "tiny":
            c = _case(None, net, log_int(1, 64), rng.randint(8, 24), rng.randint(8, 24), rng.randint(2, 20), "f32")
        elif net in ("resnet56", "resnet110", "wrn28_10"):
            f32 = net == "resnet56" and rng.random() < 0.4
            side = rng.choice([24, 28, 32, 32, 32, 36, 40])
            c = _case(None, net, log_int(4, 32 if f32 else 128), side, side, rng.choice([10, 100, rng.randint(2, 200)]),
                      "f32" if f32 else "bf16")
            c["batch"] = max(1, min(c["batch"], (32 if f32 else 128) * 1024 // (side * side)))
        else:
            top = 64 if net == "resnet34" else 32
            c = _case(None, net, log_int(2, top), 16 * rng.randint(6, 18), 16 * rng.randint(6, 18),
                      rng.choice([1000, 1000, rng.randint(20, 1000)]))
            c["batch"] = max(1, min(c["batch"], top * 224 * 224 // (c["height"] * c["width"])))
        modes = ["step", "step", "step", "three_calls", "distill"]
        # (a whole bf16 network of 50 or more layers, or a few images under batch statistics, magnifies rounding too
        # much for two correct programs to be compared at its end)
        if net == "tiny" or (net in ("resnet56", "wrn28_10", "resnet34") and c["batch"] >= 16):
            modes += ["serial", "eval"]
        c["mode"] = rng.choice(modes)
        c["modules"] = rng.choice([0, 0, rng.randint(2, 8)])
        if c["mode"] in ("step", "three_calls", "distill"):
            c["loss"] = rng.choice(["penalty", "al"])
            c["recursive"] = rng.random() < 0.2
        if c["mode"] != "eval" and c["mode"] != "distill":
            c["momentum"] = rng.choice([0.0, 0.0, 0.9])
        c["graph"] = rng.random() < 0.6
        if c["modules"] and net == "tiny":
            c["modules"] = 2
        if lp.lp_validate_desc(lp.desc_from_config(_config(c), aux_recursive=c["recursive"])) == 0:
            return c


def _config(case):
    cfg = with_modules(case["net"], case["modules"]) if case["modules"] else get_config(case["net"])
    cfg.update(dtype=case["dtype"], N=case["batch"], H=case["height"], W=case["width"], num_classes=case["classes"],
               loss=case["loss"])
    return cfg


def _parts(desc, K, recursive):
    """`which` numbers of the modules and of the AuxNets."""
    auxs = [lp.LP_REAUX(k, j) for k in range(1, K) for j in range(k)] if recursive else [lp.LP_AUX(k) for k in range(K - 1)]
    return list(range(K)), auxs


def _parameters(layout, gen, dtype):
    """Parameter values as in the middle of training: He-normal filters, affine parameters spread around 1 and 0."""
    out = []
    for _, kind, shape in layout:
        n = int(np.prod(shape))
        v = torch.randn(n, generator=gen, device="cuda")
        if kind in ("conv_w", "fc_w"):
            v *= (2.0 * shape[0] / n) ** 0.5
        elif kind == "bn_gamma":
            v = 1.0 + 0.1 * v
        else:
            v *= 0.1
        out.append(v)
    v = torch.cat(out)
    return v.to(torch.bfloat16).float() if dtype == "bf16" else v


def _view_of(h, values):
    """The handle's own copy of a parameter blob: where `values` sits in the workspace the handle was given."""
    words = h.workspace[: h.workspace.numel() // 4 * 4].view(torch.float32)
    for at in (words == values[0]).nonzero().flatten().tolist():
        if at + values.numel() <= words.numel() and torch.equal(words[at:at + values.numel()], values):
            return words[at:at + values.numel()]
    raise RuntimeError("the parameters just set are not in the workspace")


def prepare(case, seed):
    cfg = _config(case)
    K, N = cfg["K"], cfg["N"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    desc = lp.desc_from_config(cfg, aux_recursive=case["recursive"])
    h = lp.lp_create(desc)
    modules, auxs = _parts(desc, K, case["recursive"])
    values = {w: _parameters(lp.lp_param_layout(desc, w), gen, case["dtype"]) for w in modules + auxs}
    host = {w: v.cpu().numpy() for w, v in values.items()}
    for w in values:
        lp.lp_set_params(h, w, host[w])
    shapes = [lp.lp_boundary_shape_desc(desc, k) for k in range(K)]
    images = torch.randn(shapes[0], generator=gen, device="cuda").to(dt)
    labels = torch.randint(0, case["classes"], (N,), generator=gen, device="cuda", dtype=torch.int32)
    s = dict(h=h, mode=case["mode"], images=images, labels=labels, graph=None, momentum=case["momentum"],
             decay=5e-4 if case["momentum"] else 0.0, lr=_LR_PREACT if cfg["block_kind"] == "preact" else _LR)
    s["x"] = [torch.zeros(shapes[k], dtype=dt, device="cuda") for k in range(1, K)]
    s["dx"] = [None] + [torch.zeros_like(t) for t in s["x"]]
    s["kappa"] = [torch.zeros_like(t) for t in s["x"]] if case["loss"] == "al" else None
    s["loss"] = torch.zeros(K, 2, device="cuda")
    s["distill_loss"] = torch.zeros(max(K - 1, 1), device="cuda")
    s["logits"] = torch.zeros(N, case["classes"], device="cuda")
    # the penalty as a mean over the boundary's pixels: the call takes the plain sum, the scaling is the caller's
    pixels = N * max([sh[1] * sh[2] for sh in shapes[1:]] or [1])
    s["rho"] = cfg["rho"] / pixels
    if case["mode"] == "eval":
        s["out"] = {"logits": s["logits"]}
    else:
        s["out"] = {"params": [_view_of(h, values[w]) for w in modules]}
        if case["mode"] == "serial":
            s["out"]["loss"] = s["loss"][K - 1]
        else:
            s["out"].update(loss=s["loss"], x=s["x"])
            if s["kappa"] is not None:
                s["out"]["kappa"] = s["kappa"]
        if case["mode"] == "distill":
            s["out"].update(aux_params=[_view_of(h, values[w]) for w in auxs], distill_loss=s["distill_loss"])
    if case["graph"]:
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        _enqueue(s, stream.cuda_stream)          # the first call of a kind comes before any recording
        stream.synchronize()
        lp.lp_graph_begin(h, stream.cuda_stream)
        _enqueue(s, stream.cuda_stream)
        s["graph"] = lp.lp_graph_end(h, stream.cuda_stream)
        for w in values:                         # that first call was a step: back to the start
            lp.lp_set_params(h, w, host[w])
        for t in s["kappa"] or []:
            t.zero_()
    return s


def _enqueue(s, stream):
    h, mode = s["h"], s["mode"]
    if mode == "eval":
        lp.lp_forward_serial(h, s["images"], s["logits"], stream)
    elif mode == "serial":
        lp.lp_serial_fwd_bwd(h, s["images"], s["labels"], s["loss"][h.K - 1], stream)
        lp.lp_step(h, s["lr"], s["momentum"], s["decay"], 0.0, None, stream)
    elif mode == "three_calls":
        lp.lp_auxnet_forward(h, s["images"], s["x"], stream)
        lp.lp_modules_fwd_bwd_all(h, [s["images"]] + s["x"], s["labels"], s["kappa"], s["rho"], s["loss"], s["dx"], stream)
        lp.lp_step(h, s["lr"], s["momentum"], s["decay"], s["lr"] * s["rho"], s["kappa"], stream)
    else:
        lp.lp_layer_parallel_step(h, s["images"], s["x"], s["labels"], s["kappa"], s["rho"], s["loss"], s["dx"],
                                  s["lr"], s["momentum"], s["decay"], s["lr"] * s["rho"], stream)
        if mode == "distill":
            lp.lp_auxnet_distill(h, s["images"], s["x"], s["dx"], _LR_LAMBDA, _LR_AUX, None, s["distill_loss"], stream)


def run(s):
    stream = torch.cuda.current_stream().cuda_stream
    if s["graph"] is None:
        _enqueue(s, stream)
    else:
        lp.lp_graph_launch(s["h"], s["graph"], stream)
    return s["out"]


def _forward_flops(cfg, desc):
    """Multiply-adds x 2 of the convolutions: (modules, AuxNets)."""
    def out(v, r, stride, pad):
        return (v + 2 * pad - r) // stride + 1
    N, h, w = cfg["N"], cfg["H"], cfg["W"]
    fl = 0.0

    def conv(ho, wo, co, r, ci):
        return 2.0 * N * ho * wo * co * r * r * ci
    if cfg["stem_kind"] == "conv3x3":
        fl += conv(h, w, cfg["stem_channels"], 3, cfg["C_in"])
    else:
        h, w = out(h, 7, 2, 3), out(w, 7, 2, 3)
        fl += conv(h, w, cfg["stem_channels"], 7, cfg["C_in"])
        h, w = out(h, 3, 2, 1), out(w, 3, 2, 1)
    c = cfg["stem_channels"]
    for ch, blocks, stride in zip(cfg["stage_channels"], cfg["stage_blocks"], cfg["stage_stride"]):
        for b in range(blocks):
            st = stride if b == 0 else 1
            ho, wo = out(h, 3, st, 1), out(w, 3, st, 1)
            if cfg["block_kind"] == "bottleneck":
                mid = ch // 4
                fl += conv(h, w, mid, 1, c) + conv(ho, wo, mid, 3, mid) + conv(ho, wo, ch, 1, mid)
            else:
                fl += conv(ho, wo, ch, 3, c) + conv(ho, wo, ch, 3, ch)
            if st != 1 or c != ch:
                fl += conv(ho, wo, ch, 1, c)
            h, w, c = ho, wo, ch
    K = cfg["K"]
    shapes = [lp.lp_boundary_shape_desc(desc, k) for k in range(K)]
    aux = []
    for (_, hi, wi, ci), (_, ho, wo, co) in zip(shapes, shapes[1:]):
        if cfg["aux_convs"] == 1:
            aux.append(conv(ho, wo, co, 3, ci))
        else:
            s1 = 2 if hi // ho >= 2 else 1
            hid = co // cfg["aux_width_div"]
            aux.append(conv(out(hi, 3, s1, 1), out(wi, 3, s1, 1), hid, 3, ci) + conv(ho, wo, co, 3, hid))
    if desc.aux_recursive:
        return fl, sum(a * (K - 1 - j) for j, a in enumerate(aux))
    return fl, sum(aux)


def work(case):
    cfg = _config(case)
    desc = lp.desc_from_config(cfg, aux_recursive=case["recursive"])
    K = cfg["K"]
    modules, auxs = _parts(desc, K, case["recursive"])
    count = lambda ws: sum(int(np.prod(sh)) for w in ws for _, _, sh in lp.lp_param_layout(desc, w))  # noqa: E731
    p_mod, p_aux = 4.0 * count(modules), 4.0 * count(auxs)
    e = 4 if case["dtype"] == "f32" else 2
    images = float(cfg["N"] * cfg["H"] * cfg["W"] * cfg["C_in"] * e)
    bound = float(sum(np.prod(lp.lp_boundary_shape_desc(desc, k)) for k in range(1, K)) * e)
    fwd, aux = _forward_flops(cfg, desc)
    if case["mode"] == "eval":
        return {"bytes": images + p_mod + 4.0 * cfg["N"] * case["classes"], "flops": fwd}
    update = (4.0 if case["momentum"] else 2.0) * p_mod     # parameters (and momentum) read and written
    if case["mode"] == "serial":
        return {"bytes": images + update, "flops": 3.0 * fwd}
    bytes_ = images + update + p_aux + 2.0 * bound          # x_k and dx_k written
    if case["loss"] == "al":
        bytes_ += 2.0 * bound                               # multipliers read and written
    flops = 3.0 * fwd + aux
    if case["mode"] == "distill":
        bytes_ += p_aux                                     # AuxNet parameters written too
        flops += 2.0 * aux
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """fp32: sums in another order.  bf16: once a sum is taken in another order a stored activation rounds to its
    neighbour, and after a few layers all of them differ by rounding.  Between two sets of convolution kernels
    (tensor cores, CUDA cores) AuxNet outputs then differ by 0.7 %, residuals and multipliers by 1.2 %, the logits of
    a whole network by 2.1 %, updated parameters by 0.1 to 0.5 %.  The gradients themselves, dx_k among them, differ by
    5 to 15 % for nine-block modules (ReLU masks flip) and are seen through the updated parameters.  fp32: with the
    images changed by one rounding, parameters differ by 2e-5 after two passes."""
    if case["dtype"] == "f32":
        return {"rel": 1e-4, "max": 2e-3}
    if case["mode"] == "eval":
        return {"rel": 3e-2, "max": 0.5}
    return {"rel": 3e-2 if case["loss"] == "al" else 2e-2, "max": 0.3}
