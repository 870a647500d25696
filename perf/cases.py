"""The framework's work, case by case: forward layers, gradients, training-mode normalisation,
the RGB stem and the whole backbone, through the public entry points of the Python package.

A case is a dict of plain values.  `kind` says which calls one pass makes:

  conv      one quaternion convolution with its epilogue (`quan.qconv2d`): bf16 or fp32
            tensors, full or separable form, optionally a residual, ReLU / SiLU / none
  grad      the two gradients of a convolution's backward pass
            (`quan.qconv2d_backward_data`, `quan.qconv2d_backward_weight`)
  step      one layer's share of a training step: the convolution without an epilogue, then
            both gradients
  iqbn      training-mode IQBN: batch statistics, normalisation and activation
            (`quan.iqbn_train`)
  stem_rgb  the 7x7/2 stem with its 3x3/2 max pool from fp32 RGB images, the Poincare
            mapping fused (`quan.quan_qconv2d_maxpool_rgb_fwd`)
  backbone  a whole forward pass of the ResNet-18-style backbone (`BackboneRunner.step`, as
            the benchmark configures it)

Values follow the package's recipe: activations and output gradients N(0, 1), letters
N(0, 1 / (C_in kh kw)), IQBN scale U(0.5, 1.5), shift and bias N(0, 0.1^2), RGB U(0, 1).
"""
import math

import numpy as np
import torch

from paper_2509_05512_gb300 import backbone, inputs, quan

ACT = {"none": quan.QUAN_ACT_NONE, "relu": quan.QUAN_ACT_RELU, "silu": quan.QUAN_ACT_SILU}

# Work of the largest listed layer that runs on the tensor cores (the 56 x 56 convolution),
# and of the largest that does not, per form of call: a drawn case stays below.
MAX_TC_FLOPS = 2.3e11
MAX_NARROW_FLOPS = 1.3e9


def _conv(kind, N, H, W, Cin, Cout, k, stride, **extra):
    case = {"kind": kind, "N": N, "H": H, "W": W, "Cin": Cin, "Cout": Cout, "k": k,
            "stride": stride, "pad": k // 2, "dtype": "bf16", "form": "full", "act": "none",
            "bias": False, "iqbn": False, "residual": False}
    case.update(extra)
    return case


def listed():
    return [
        # the smallest call of the package's own configurations: one fp32 layer with a bias on
        # 8 x 8 images, as in a unit test or a first experiment; latency and the launch count
        dict(_conv("conv", 2, 8, 8, 16, 16, 3, 1, dtype="f32", bias=True), name="f32_small"),
        # an fp32 layer of ordinary size: evaluation at full precision, batch 8
        dict(_conv("conv", 8, 32, 32, 64, 64, 3, 1, dtype="f32", iqbn=True, act="relu"),
             name="f32_layer"),
        # the CIFAR-shaped layer at inference
        dict(_conv("conv", 128, 32, 32, 64, 64, 3, 1, iqbn=True, act="relu"), name="cifar_fwd"),
        # the ImageNet stage layer at inference, the benchmark's compute-bound layer
        dict(_conv("conv", 64, 56, 56, 256, 256, 3, 1, iqbn=True, act="relu"),
             name="imagenet_fwd"),
        # the detection neck's 1x1 layer with the detector's SiLU (640-pixel input, stride 8)
        dict(_conv("conv", 16, 80, 80, 512, 1024, 1, 1, iqbn=True, act="silu"),
             name="neck_pointwise"),
        # the backward pass of the CIFAR-shaped layer
        dict(_conv("grad", 128, 32, 32, 64, 64, 3, 1), name="cifar_grad"),
        # the backward pass of the ImageNet downsampling layer (stride 2)
        dict(_conv("grad", 64, 56, 56, 256, 512, 3, 2), name="imagenet_down_grad"),
        # a training step of a separable layer (the paper's reduced form)
        dict(_conv("step", 32, 28, 28, 128, 128, 3, 1, form="sep"), name="sep_step"),
        # a training step of a narrow layer on odd-sized images: a small detector's or CIFAR
        # network's widths, channel counts off the tensor-core grid
        dict(_conv("step", 16, 45, 37, 24, 40, 3, 1), name="narrow_step"),
        # training-mode IQBN + ReLU of the ImageNet stage activation
        {"kind": "iqbn", "N": 64, "H": 56, "W": 56, "C": 256, "act": "relu",
         "name": "iqbn_train"},
        # the camera end of the backbone: RGB images to pooled quaternion features
        {"kind": "stem_rgb", "N": 64, "H": 224, "W": 224, "act": "relu", "name": "stem_rgb"},
        # a whole inference call, the benchmark's default workload
        {"kind": "backbone", "N": 256, "H": 224, "name": "backbone"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit_batch(rng, case, lo, hi, cap, passes):
    """A batch in [lo, hi], log-spread, whose work stays below cap."""
    per = passes * _conv_flops(dict(case, N=1))
    return max(1, min(_log(rng, lo, hi), int(cap / per)))


def draw(rng):
    what = rng.choice(["f32", "conv", "conv", "pointwise", "grad", "grad", "sep", "narrow",
                       "narrow", "iqbn", "stem_rgb", "backbone"])
    act = rng.choice(["none", "relu", "relu", "silu"])
    if what == "f32":
        case = _conv("conv", 1, _log(rng, 5, 40), _log(rng, 5, 40), 4 * rng.randint(1, 20),
                     4 * rng.randint(1, 20), rng.choice([1, 3, 3, 5]), rng.choice([1, 1, 2]),
                     dtype="f32", bias=rng.random() < 0.5, iqbn=rng.random() < 0.5, act=act)
        case["N"] = _fit_batch(rng, case, 1, 16, 6.0e8, 1)
    elif what == "narrow":
        case = _conv("step", 1, _log(rng, 7, 60), _log(rng, 7, 60), 4 * rng.randint(1, 15),
                     4 * rng.randint(1, 15), rng.choice([1, 3, 3]), rng.choice([1, 1, 2]))
        case["N"] = _fit_batch(rng, case, 1, 64, MAX_NARROW_FLOPS, 3)
    elif what == "iqbn":
        C = rng.choice([rng.randint(2, 15) * 4, rng.randint(8, 64) * 8, rng.randint(1, 8) * 64])
        H, W = _log(rng, 7, 112), _log(rng, 7, 112)
        N = max(1, min(_log(rng, 1, 256), 51_000_000 // (H * W * C)))
        case = {"kind": "iqbn", "N": N, "H": H, "W": W, "C": C, "act": act}
    elif what == "stem_rgb":
        case = {"kind": "stem_rgb", "N": _log(rng, 1, 64), "H": rng.randint(64, 224),
                "W": 32 * rng.randint(2, 7), "act": act}
    elif what == "backbone":
        case = {"kind": "backbone", "N": _log(rng, 1, 256), "H": 32 * rng.randint(3, 7)}
    else:
        if what == "pointwise":
            case = _conv("conv", 1, _log(rng, 10, 80), _log(rng, 10, 80),
                         64 * rng.randint(1, 8), 64 * rng.randint(1, 16), 1,
                         rng.choice([1, 1, 2]), iqbn=True, act=act)
        elif what == "conv":
            case = _conv("conv", 1, _log(rng, 7, 80), _log(rng, 7, 80), 64 * rng.randint(1, 8),
                         64 * rng.randint(1, 8), 3, rng.choice([1, 1, 2]), iqbn=True, act=act,
                         residual=rng.random() < 0.3)
        else:
            case = _conv("step" if what == "sep" else "grad", 1, _log(rng, 7, 64),
                         _log(rng, 7, 64), 64 * rng.randint(1, 6),
                         64 * rng.choice([1, 2, 3, 4, 8]), rng.choice([1, 3, 3]),
                         rng.choice([1, 1, 2]), form="sep" if what == "sep" else "full")
        passes = {"conv": 1, "grad": 2, "step": 3}[case["kind"]]
        cap = 4.0e10 if what == "sep" else MAX_TC_FLOPS
        case["N"] = _fit_batch(rng, case, 1, 128, cap, passes)
    return case


# ------------------------------------------------------------------ sizes and work

def _out_hw(case):
    k, s, p = case["k"], case["stride"], case["pad"]
    return quan.out_size(case["H"], k, s, p), quan.out_size(case["W"], k, s, p)


def _conv_flops(case):
    Ho, Wo = _out_hw(case)
    form = 4 if case["form"] == "sep" else 1  # Eq. 7 keeps a quarter of the products
    return (2.0 * case["N"] * Ho * Wo * case["Cout"] * case["Cin"] * case["k"] ** 2) / form


def _backbone_layers(case):
    return inputs.backbone_layers(N=case["N"], H=case["H"])


def work(case):
    kind = case["kind"]
    if kind == "iqbn":
        n = case["N"] * case["H"] * case["W"] * case["C"]
        return {"bytes": 4 * n + 16 * case["C"], "flops": 8 * n}
    if kind == "stem_rgb":
        N, H, W = case["N"], case["H"], case["W"]
        Ho, Wo = quan.out_size(H, 7, 2, 3), quan.out_size(W, 7, 2, 3)
        Hp, Wp = quan.out_size(Ho, 3, 2, 1), quan.out_size(Wo, 3, 2, 1)
        return {"bytes": 12 * N * H * W + 2 * N * Hp * Wp * 64 + 2 * 49 * 64 + 8 * 64,
                "flops": 2 * N * Ho * Wo * 64 * 4 * 49}
    if kind == "backbone":
        layers = _backbone_layers(case)
        last = layers[-1].spec
        convs = [L.spec for L in layers if L.kind == "conv"]
        return {"bytes": 8 * case["N"] * case["H"] ** 2 + 2 * case["N"] * last.Ho * last.Wo *
                last.Cout + sum(s.Cout * s.Cin * s.kh * s.kw / 2 + 8 * s.Cout for s in convs),
                "flops": sum(s.flops for s in convs)}
    e = 4 if case["dtype"] == "f32" else 2
    Ho, Wo = _out_hw(case)
    H, W = (Ho, Wo) if case["k"] == 1 else (case["H"], case["W"])  # 1x1: the sampled pixels
    nx, ny = case["N"] * H * W * case["Cin"], case["N"] * Ho * Wo * case["Cout"]
    nw = case["Cout"] * case["Cin"] * case["k"] ** 2 // 4
    nx_all = case["N"] * case["H"] * case["W"] * case["Cin"]
    flops = _conv_flops(case)
    if kind == "conv":
        vectors = 4 * case["Cout"] * (int(case["bias"]) + 2 * int(case["iqbn"]))
        return {"bytes": e * (nx + ny * (2 if case["residual"] else 1) + nw) + vectors,
                "flops": flops}
    # gradients: x, dy and the letters read, dx (bf16) and the letters' gradients (fp32) written
    grads = {"bytes": e * (nx + ny + nw + nx_all) + 4 * nw, "flops": 2 * flops}
    if kind == "grad":
        return grads
    return {"bytes": grads["bytes"] + e * ny, "flops": 3 * flops}


# ------------------------------------------------------------------ inputs

def _letters(gen, case, dtype):
    shape = (case["Cout"] // 4, case["k"], case["k"], case["Cin"] // 4)
    std = 1.0 / math.sqrt(case["Cin"] * case["k"] ** 2)
    return [(torch.randn(shape, generator=gen, device="cuda") * std).to(dtype)
            for _ in range(4)]


def _vectors(gen, C):
    return (torch.rand(C, generator=gen, device="cuda") + 0.5,
            torch.randn(C, generator=gen, device="cuda") * 0.1)


def prepare(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    state = {"case": case}
    if kind == "iqbn":
        x = torch.randn((case["N"], case["H"], case["W"], case["C"]), generator=gen,
                        device="cuda")
        gamma, beta = _vectors(gen, case["C"])
        state.update(x=x.to(torch.bfloat16), gamma=gamma, beta=beta)
    elif kind == "stem_rgb":
        stem = {"Cin": 4, "Cout": 64, "k": 7}
        state["rgb"] = torch.rand((case["N"], case["H"], case["W"], 3), generator=gen,
                                  device="cuda")
        state["w"] = _letters(gen, stem, torch.bfloat16)
        state["scale"], state["shift"] = _vectors(gen, 64)
    elif kind == "backbone":
        x = torch.rand((case["N"], case["H"], case["H"], 4), generator=gen, device="cuda")
        bits = (2.0 * x - 1.0).to(torch.bfloat16).view(torch.int16).cpu().numpy()
        state["runner"] = backbone.BackboneRunner(
            torch, quan, inputs, N=case["N"], H=case["H"], seed=seed,
            x_bits=bits.view(np.uint16), fuse_stem_pool=True, overlap_shortcuts=True,
            split_k=True)
        # the stream the program runs the network on (the shortcuts fork from and join it)
        state["stream"] = torch.cuda.Stream()
    else:
        dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        Ho, Wo = _out_hw(case)
        yshape = (case["N"], Ho, Wo, case["Cout"])
        state["x"] = torch.randn((case["N"], case["H"], case["W"], case["Cin"]), generator=gen,
                                 device="cuda").to(dtype)
        state["w"] = _letters(gen, case, dtype)
        state["bias"] = (torch.randn(case["Cout"], generator=gen, device="cuda") * 0.1
                         if case["bias"] else None)
        state["scale"], state["shift"] = (_vectors(gen, case["Cout"]) if case["iqbn"]
                                          else (None, None))
        state["residual"] = (torch.randn(yshape, generator=gen, device="cuda").to(dtype)
                             if case["residual"] else None)
        if kind != "conv":
            state["dy"] = torch.randn(yshape, generator=gen, device="cuda").to(dtype)
    return state


# ------------------------------------------------------------------ one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "iqbn":
        return quan.iqbn_train(state["x"], state["gamma"], state["beta"], act=ACT[case["act"]])
    if kind == "stem_rgb":
        rgb = state["rgb"]
        N, H, W, _ = rgb.shape
        Hp = quan.out_size(quan.out_size(H, 7, 2, 3), 3, 2, 1)
        Wp = quan.out_size(quan.out_size(W, 7, 2, 3), 3, 2, 1)
        out = torch.empty((N, Hp, Wp, 64), dtype=torch.bfloat16, device=rgb.device)
        quan.quan_qconv2d_maxpool_rgb_fwd(rgb, *state["w"], None, state["scale"],
                                          state["shift"], N, H, W, 64, 7, 7, 2, 3,
                                          ACT[case["act"]], out)
        return out
    if kind == "backbone":
        runner, stream, caller = state["runner"], state["stream"], torch.cuda.current_stream()
        stream.wait_stream(caller)
        runner.step(stream.cuda_stream)
        caller.wait_stream(stream)
        return runner.output
    x, w = state["x"], state["w"]
    k, geo, sep = case["k"], {"stride": case["stride"], "pad": case["pad"]}, case["form"] == "sep"
    if kind == "conv":
        return quan.qconv2d(x, *w, **geo, bias=state["bias"], scale=state["scale"],
                            shift=state["shift"], act=ACT[case["act"]],
                            residual=state["residual"], separable=sep)
    out = []
    if kind == "step":
        out.append(quan.qconv2d(x, *w, **geo, separable=sep))
    dy = state["dy"]
    out.append(quan.qconv2d_backward_data(dy, *w, H=case["H"], W=case["W"], **geo,
                                          separable=sep))
    out.extend(quan.qconv2d_backward_weight(x, dy, kh=k, kw=k, **geo, separable=sep))
    return out


# ------------------------------------------------------------------ tolerance and exact values

def tolerance(case):
    # bf16 outputs rounded once from fp32 sums; the gradients' letters and the fp32 layers are
    # fp32 sums; every layer of the backbone rounds its activations to bf16.  Seen against
    # exact(): bf16 1.66e-3 and 3.9e-3 (half an ulp), fp32 4e-7 to 8e-7 and 4e-6, the
    # backbone 5.4e-3; about four times that
    if case["kind"] == "backbone":
        return {"rel": 2.0e-2, "max": 2.0e-1}
    if case["kind"] == "conv" and case["dtype"] == "f32":
        return {"rel": 3.0e-6, "max": 1.6e-5}
    return {"rel": 6.6e-3, "max": 1.6e-2}


# Output component q takes input component p through letter q xor p (Eq. 5), negative where
# FULL_NEG says so; the separable form (Eq. 7) takes input component p through letter p.
FULL_NEG = {(0, 1), (0, 2), (0, 3), (1, 2), (2, 3), (3, 1)}
SEP_NEG = {(0, 1), (0, 2), (0, 3), (1, 3), (2, 1), (3, 2)}


def _sign(q, p, sep):
    return -1.0 if (q, p) in (SEP_NEG if sep else FULL_NEG) else 1.0


def _real_weight(w, sep):
    """The real weight [Cout, Cin, k, k] of the block matrix, fp64."""
    w = [t.double().permute(0, 3, 1, 2) for t in w]
    rows = [torch.cat([_sign(q, p, sep) * w[p if sep else q ^ p] for p in range(4)], dim=1)
            for q in range(4)]
    return torch.cat(rows, dim=0).contiguous()


def _act64(z, act):
    if act == "relu":
        return torch.relu(z)
    if act == "silu":
        return z * torch.sigmoid(z)
    return z


def _nhwc(t):
    return t.permute(0, 2, 3, 1).contiguous()


def _nchw(t):
    return t.double().permute(0, 3, 1, 2).contiguous()


def _letter_grads(dreal, sep):
    """Gradients of the four letters from the real weight's gradient [Cout, Cin, k, k]."""
    Qo, Qi = dreal.shape[0] // 4, dreal.shape[1] // 4
    out = []
    for L in range(4):
        g = 0.0
        for q in range(4):
            p = L if sep else q ^ L
            g = g + _sign(q, p, sep) * dreal[q * Qo:(q + 1) * Qo, p * Qi:(p + 1) * Qi]
        out.append(g.permute(0, 2, 3, 1).contiguous())
    return out


def _exact_backbone(state):
    import torch.nn.functional as F
    runner = state["runner"]
    outs = []
    for s0 in range(0, runner.N, 32):  # 32 images at a time bound the fp64 activations
        feats = []
        for i, L in enumerate(runner.layers):
            src = _nchw(runner.x[s0:s0 + 32]) if L.src == -1 else feats[L.src]
            if L.kind == "maxpool":
                feats.append(F.max_pool2d(src, L.k, L.stride, L.pad))
                continue
            prm = runner.params[i]
            z = F.conv2d(src, _real_weight(prm["w"], False), stride=L.spec.stride,
                         padding=L.spec.pad)
            z = z * prm["scale"].double().view(1, -1, 1, 1) + \
                prm["shift"].double().view(1, -1, 1, 1)
            if L.res is not None:
                z = z + feats[L.res]
            feats.append(torch.relu(z) if L.spec.act == quan.QUAN_ACT_RELU else z)
        outs.append(_nhwc(feats[-1]))
    return torch.cat(outs)


def exact(case, seed):
    import torch.nn.functional as F
    state = prepare(case, seed)
    kind = case["kind"]
    if kind == "iqbn":
        x = state["x"].double()
        mean = x.mean(dim=(0, 1, 2))
        var = ((x - mean) ** 2).mean(dim=(0, 1, 2))
        z = state["gamma"].double() * (x - mean) / torch.sqrt(var + 1e-5) + state["beta"].double()
        return _act64(z, case["act"]), mean, var
    if kind == "backbone":
        return _exact_backbone(state)
    if kind == "stem_rgb":
        c = state["rgb"].double()
        n2 = (c * c).sum(dim=-1, keepdim=True)
        # the quaternion pixels are bf16 tensors in the package's data model
        x = (torch.cat([1.0 - n2, 2.0 * c], dim=-1) / (1.0 + n2)).to(torch.bfloat16)
        z = F.conv2d(_nchw(x), _real_weight(state["w"], False), stride=2, padding=3)
        z = z * state["scale"].double().view(1, -1, 1, 1) + \
            state["shift"].double().view(1, -1, 1, 1)
        return _nhwc(F.max_pool2d(_act64(z, case["act"]), 3, 2, 1))
    sep, geo = case["form"] == "sep", {"stride": case["stride"], "padding": case["pad"]}
    w = _real_weight(state["w"], sep)
    out = []
    if kind in ("conv", "step"):
        z = F.conv2d(_nchw(state["x"]), w, **geo)
        if kind == "conv":
            if state["bias"] is not None:
                z = z + state["bias"].double().view(1, -1, 1, 1)
            if state["scale"] is not None:
                z = z * state["scale"].double().view(1, -1, 1, 1) + \
                    state["shift"].double().view(1, -1, 1, 1)
            if state["residual"] is not None:
                z = z + _nchw(state["residual"])
            return _nhwc(_act64(z, case["act"]))
        out.append(_nhwc(z))
    dy, x = _nchw(state["dy"]), _nchw(state["x"])
    out.append(_nhwc(torch.nn.grad.conv2d_input(x.shape, w, dy, **geo)))
    out.extend(_letter_grads(torch.nn.grad.conv2d_weight(x, w.shape, dy, **geo), sep))
    return out
