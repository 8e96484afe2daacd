"""The work that a user of this library has it do, as cases that can be timed and compared.

Every case is one pass through the public entry points: a single pointwise layer, a network's
pointwise layers as a stack (with and without CUDA graph replay), the strided / residual form,
the 3x3 layers, a call on host buffers and the latency-constrained projection.  Shapes are those
of alcs_workloads (MobileNetV1 and ResNet pointwise layers, ResNet-18 3x3 layers, the 512 -> 512
sweep) or generic; weights, masks and activations follow the same distributions, made on the GPU
from the seed.

  listed()            the named cases
  draw(rng)           one more case of the same ranges
  prepare(case, seed) inputs and handles a program has in hand before the call
  run(state)          one pass; returns everything it computes
  work(case)          bytes and floating-point operations the pass cannot do without
  tolerance(case)     how far another correct implementation may be off
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_00170_b200 as A
from alcs_workloads.conv2d import RESNET18_3X3
from alcs_workloads.layers import MOBILENET_V1_PW, RESNET50_BOTTLENECK_PW

# Every fixed choice below (seeds of the distributions, sizes) is in the case; nothing is read from disk.


def listed():
    return [
        # The smallest call: one layer of one image, as a latency-bound program makes it.
        dict(name="single_b1", kind="layer", dtype="f32", g=4, n=1, cin=64, cout=128, h=56, w=56, sparsity=0.7,
             rows="uniform", stride=1, residual=False, relu=True, bias=True, y_f32=False),
        # The paper's own setting: the pointwise layers of MobileNetV1 for one image, replayed as a graph.
        dict(name="mbv1_b1_graph", kind="stack", net="mobilenet_v1", dtype="f32", g=4, n=1, res=224,
             sparsity_lo=0.8, sparsity_hi=0.8, graph=True),
        # The repository's headline workload: the same layers for a batch, sparsity differing by layer.
        dict(name="mbv1_b64", kind="stack", net="mobilenet_v1", dtype="f32", g=4, n=64, res=224,
             sparsity_lo=0.6, sparsity_hi=0.9, graph=False),
        # Half-precision batch inference: ResNet-50's bottleneck pointwise layers.
        dict(name="rn50_b32_f16", kind="stack", net="resnet50", dtype="f16", g=8, n=32, res=224,
             sparsity_lo=0.75, sparsity_hi=0.75, graph=False),
        # A down-sampling shortcut of a ResNet in bfloat16: stride 2, no activation of its own.
        dict(name="shortcut_s2_bf16", kind="layer", dtype="bf16", g=8, n=32, cin=256, cout=512, h=56, w=56,
             sparsity=0.75, rows="uniform", stride=2, residual=False, relu=False, bias=True, y_f32=False),
        # The last layer of a bottleneck: 7x7 images, the shortcut added before the activation.
        dict(name="expand_residual_f16", kind="layer", dtype="f16", g=8, n=32, cin=512, cout=2048, h=7, w=7,
             sparsity=0.75, rows="uniform", stride=1, residual=True, relu=True, bias=True, y_f32=False),
        # Unstructured pruning (g = 1), large batch: the weights nobody grouped.
        dict(name="unstructured_b256", kind="layer", dtype="f32", g=1, n=256, cin=512, cout=512, h=14, w=14,
             sparsity=0.9, rows="uniform", stride=1, residual=False, relu=True, bias=True, y_f32=False),
        # Skewed rows, as global magnitude pruning leaves them: kept blocks per row follow a Zipf law.
        dict(name="zipf_b256", kind="layer", dtype="f32", g=4, n=256, cin=512, cout=512, h=14, w=14,
             sparsity=0.0, rows="zipf", stride=1, residual=False, relu=True, bias=True, y_f32=False),
        # General convolution: the distinct 3x3 layers of ResNet-18, one call each.
        dict(name="rn18_3x3_b32", kind="conv2d", layers="resnet18", g=4, n=32, sparsity=0.7,
             cin=0, cout=0, h=0, w=0, k=3, stride=0, pad=1),
        # Odd sizes: a channel count that is no multiple of anything, images of 17 x 23 pixels.
        dict(name="ragged_f32", kind="layer", dtype="f32", g=4, n=5, cin=100, cout=150, h=17, w=23, sparsity=0.6,
             rows="uniform", stride=1, residual=False, relu=False, bias=True, y_f32=False),
        # Activations that live in (pinned) host memory, results read back there.
        dict(name="host_b16", kind="host", dtype="f32", g=4, n=16, cin=256, cout=512, h=14, w=14, sparsity=0.8),
        # One projection step of the pruning loop: all groups of MobileNetV1's pointwise layers onto a
        # latency budget, masks and projected weights written.
        dict(name="project_mbv1", kind="project", net="mobilenet_v1", g=4, budget=0.5),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case.  Single layers are drawn most often, then stacks, 3x3 layers, host calls, projections."""
    kind = rng.choice(["layer", "layer", "layer", "layer", "stack", "stack", "conv2d", "conv2d", "host", "project"])
    if kind == "stack":
        net = rng.choice(["mobilenet_v1", "resnet50"])
        n = _log_int(rng, 1, 64 if net == "mobilenet_v1" else 32)
        lo = round(rng.uniform(0.5, 0.85), 3)
        dtype, g = ("f32", 4) if net == "mobilenet_v1" else (rng.choice(["f16", "f16", "bf16"]), 8)
        return dict(kind="stack", net=net, dtype=dtype, g=g, n=n, res=rng.choice([128, 160, 192, 224]),
                    sparsity_lo=lo, sparsity_hi=round(rng.uniform(lo, 0.95), 3), graph=n <= 8 and rng.random() < 0.6)
    if kind == "conv2d":
        cin, cout, s, stride = rng.choice(RESNET18_3X3)
        cin = max(16, int(cin * rng.uniform(0.6, 1.0)))
        return dict(kind="conv2d", layers="one", g=rng.choice([4, 4, 8]), n=_log_int(rng, 1, 32),
                    sparsity=round(rng.uniform(0.5, 0.9), 3), cin=cin, cout=cout, h=s + rng.choice([0, 0, 1, 3]), w=s,
                    k=3, stride=stride, pad=1)
    if kind == "host":
        s = rng.choice([7, 14, 14, 28, 20])
        return dict(kind="host", dtype=rng.choice(["f32", "f32", "f16"]), g=rng.choice([4, 8]), n=_log_int(rng, 1, 32),
                    cin=_log_int(rng, 32, 512), cout=_log_int(rng, 32, 1024 if s < 20 else 512), h=s, w=s,
                    sparsity=round(rng.uniform(0.5, 0.95), 3))
    if kind == "project":
        return dict(kind="project", net=rng.choice(["mobilenet_v1", "resnet50"]), g=rng.choice([1, 4, 4, 8]),
                    budget=round(rng.uniform(0.2, 0.9), 3))
    # a single layer: sizes over their logarithm, bounded by the largest listed layer
    dtype = rng.choice(["f32", "f32", "f32", "f16", "bf16"])
    g = rng.choice([1, 4, 4, 8, 16]) if dtype == "f32" else rng.choice([8, 8, 16])
    while True:
        n, cin, cout = _log_int(rng, 1, 256), _log_int(rng, 16, 2048), _log_int(rng, 16, 2048)
        s = rng.choice([7, 7, 14, 14, 28, 56, 112, 0])
        h, w = (s, s) if s else (rng.randint(3, 60), rng.randint(3, 60))
        q = n * h * w
        if q * (cin + cout) <= 100e6 and q * cin * cout <= 13.2e9 and q >= 49:
            break
    special = dtype != "f32" or rng.random() < 0.2
    return dict(kind="layer", dtype=dtype, g=g, n=n, cin=cin, cout=cout, h=h, w=w, sparsity=round(rng.uniform(0.5, 0.95), 3),
                rows="zipf" if dtype == "f32" and g == 4 and rng.random() < 0.15 else "uniform",
                stride=2 if special and rng.random() < 0.35 else 1, residual=special and rng.random() < 0.4,
                relu=rng.random() < 0.7, bias=rng.random() < 0.9, y_f32=dtype != "f32" and rng.random() < 0.2)


# ---------------------------------------------------------------------------------------------
# The layers behind a case

def _up(a, b):
    return -(-a // b)


def _net_layers(case):
    """(cin, cout, h) of every pointwise layer of the network at the case's input resolution."""
    table = MOBILENET_V1_PW if case["net"] == "mobilenet_v1" else RESNET50_BOTTLENECK_PW
    return [(ci, co, max(1, _up(s * case.get("res", 224), 224))) for ci, co, s in table]


def _sparsities(case, n_layers):
    """Per-layer sparsity: spread evenly over [lo, hi] in a fixed scrambled order (a property of the case)."""
    lo, hi = case["sparsity_lo"], case["sparsity_hi"]
    return [lo + (hi - lo) * ((i * 0.6180339887498949) % 1.0) for i in range(n_layers)]


def _conv_layers(case):
    """(cin, cout, h, w, stride) of every call of a conv2d case."""
    if case["layers"] == "resnet18":
        return [(ci, co, s, s, st) for ci, co, s, st in RESNET18_3X3]
    return [(case["cin"], case["cout"], case["h"], case["w"], case["stride"])]


def _kept(rows, cols, sparsity):
    return rows * cols - min(rows * cols, int(round(sparsity * rows * cols)))


_ZIPF_A = 1.2


def _zipf_pmf(cin):
    p = np.arange(1, cin + 1, dtype=np.float64) ** -_ZIPF_A
    return p / p.sum()


_TORCH = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_ELT = {"f32": 4, "f16": 2, "bf16": 2}


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _mask(rows, cols, sparsity, kind, gen, seed):
    """Block mask [rows, cols]: an exact number of blocks dropped, or Zipf-distributed row lengths."""
    u = torch.rand(rows, cols, generator=gen, device="cuda")
    if kind == "zipf":
        counts = 1 + np.random.RandomState(seed & 0x7fffffff).choice(cols, size=rows, p=_zipf_pmf(cols))
        rank = u.argsort(dim=1).argsort(dim=1)
        m = rank < torch.from_numpy(counts).to("cuda")[:, None]
    else:
        m = torch.zeros(rows * cols, dtype=torch.bool, device="cuda")
        m[u.reshape(-1).argsort()[:_kept(rows, cols, sparsity)]] = True
    return m.reshape(rows, cols).to(torch.uint8).cpu().numpy()


def _packed(cout, cols, g, dtype, sparsity, kind, gen, seed):
    """Packed weights N(0, 1/cols) on the GPU, as a program keeps them."""
    w = (torch.randn(cout, cols, generator=gen, device="cuda") * cols ** -0.5).to(_TORCH[dtype]).cpu()
    m = _mask(_up(cout, g), cols, sparsity, kind, gen, seed)
    if dtype == "bf16":
        p = A.alcs_pack(w.view(torch.int16).numpy().view(np.uint16), m, g, bf16=True)
    else:
        p = A.alcs_pack(w.numpy(), m, g)
    return A.alcs_packed_upload(p, torch.cuda.current_device())


def _acts(shape, dtype, gen):
    """Activations behind a ReLU: U[0, 1) in fp32, |N(0, 1)| in the 16-bit types."""
    if dtype == "f32":
        return torch.rand(shape, generator=gen, device="cuda")
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).abs_().to(_TORCH[dtype])


def _bias(cout, gen):
    return torch.randn(cout, generator=gen, device="cuda") * 0.1


def prepare(case, seed):
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "layer":
        n, g, dt, s = case["n"], case["g"], case["dtype"], case["stride"]
        oh, ow = _up(case["h"], s), _up(case["w"], s)
        ydt = torch.float32 if case["y_f32"] else _TORCH[dt]
        st = dict(case=case, w=_packed(case["cout"], case["cin"], g, dt, case["sparsity"], case["rows"], gen, seed))
        st["x"] = _acts((n, case["cin"], case["h"] * case["w"]), dt, gen)
        st["y"] = torch.empty((n, case["cout"], oh * ow), dtype=ydt, device="cuda")
        st["bias"] = _bias(case["cout"], gen) if case["bias"] else None
        st["res"] = torch.randn((n, case["cout"], oh * ow), generator=gen, device="cuda").to(ydt) if case["residual"] else None
        st["flags"] = (A.ALCS_RELU if case["relu"] else 0) | (A.ALCS_Y_F32 if case["y_f32"] else 0)
        return st
    if kind == "stack":
        layers, table = [], _net_layers(case)
        for (ci, co, s), sp in zip(table, _sparsities(case, len(table))):
            layers.append(dict(w=_packed(co, ci, case["g"], case["dtype"], sp, "uniform", gen, seed),
                               x=_acts((case["n"], ci, s * s), case["dtype"], gen),
                               y=torch.empty((case["n"], co, s * s), dtype=_TORCH[case["dtype"]], device="cuda"),
                               n=case["n"], h=s, wd=s, bias=_bias(co, gen), flags=A.ALCS_RELU))
        torch.cuda.synchronize()
        return dict(case=case, stack=A.alcs_stack_create(layers, A.ALCS_STACK_GRAPH if case["graph"] else 0),
                    y=[L["y"] for L in layers])
    if kind == "conv2d":
        k, pad, calls = case["k"], case["pad"], []
        for ci, co, h, w, s in _conv_layers(case):
            oh, ow = (h + 2 * pad - k) // s + 1, (w + 2 * pad - k) // s + 1
            calls.append(dict(w=_packed(co, ci * k * k, case["g"], "f32", case["sparsity"], "uniform", gen, seed),
                              x=_acts((case["n"], ci, h, w), "f32", gen),
                              y=torch.empty((case["n"], co, oh, ow), device="cuda"), bias=_bias(co, gen), ci=ci, h=h, wd=w, s=s))
        return dict(case=case, calls=calls)
    if kind == "host":
        n, ci, co, hw, dt = case["n"], case["cin"], case["cout"], case["h"] * case["w"], case["dtype"]
        p = _packed(co, ci, case["g"], dt, case["sparsity"], "uniform", gen, seed)
        x = torch.empty((n, ci, hw), dtype=_TORCH[dt], pin_memory=True)
        x.copy_(_acts((n, ci, hw), dt, gen))
        b = torch.empty(co, pin_memory=True)
        b.copy_(_bias(co, gen))
        ws = torch.empty(A.alcs_spconv1x1_host_workspace(p, n, case["h"], case["w"], A.ALCS_RELU), dtype=torch.uint8, device="cuda")
        return dict(case=case, w=p, x=x, bias=b, ws=ws, y=torch.empty((n, co, hw), dtype=_TORCH[dt], pin_memory=True))
    if kind == "project":
        us = [torch.randn(co, ci, generator=gen, device="cuda") * (ci ** -0.5) for ci, co, _ in _net_layers(case)]
        tabs = []
        for (ci, co, s), u in zip(_net_layers(case), us):      # run time against kept weights: a floor, then linear, 11 knots
            n = _up(co, case["g"]) * ci * case["g"]
            ks = [n * i // 10 for i in range(11)]
            fl = 5.0 + 1e-5 * s * s * (ci + co)
            tabs.append((np.array(ks, np.int64), np.array([max(fl, 2.0 + 60.0 * i / 10 * n / 262144) + 0.1 * i for i in range(11)])))
        lo, hi = 20.0 + sum(t[0] for _, t in tabs), 20.0 + sum(t[-1] for _, t in tabs)
        total = sum(_up(u.shape[0], case["g"]) * u.shape[1] for u in us)
        return dict(case=case, u=us, tabs=tabs, tau=20.0, budget=lo + case["budget"] * (hi - lo), eps=1e-3 * (hi - lo),
                    mask=torch.empty(total, dtype=torch.uint8, device="cuda"), out=[torch.empty_like(u) for u in us])
    raise ValueError(kind)


def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    if kind == "layer":
        if case["stride"] == 1 and not case["residual"]:
            A.alcs_spconv1x1(state["w"], state["x"], state["y"], case["n"], case["h"], case["w"], state["bias"], state["flags"], stream)
        else:
            A.alcs_spconv1x1_ex(state["w"], state["x"], state["y"], case["n"], case["h"], case["w"], case["stride"], state["bias"],
                                state["res"], state["flags"], stream)
        return state["y"]
    if kind == "stack":
        A.alcs_stack_run(state["stack"], stream)
        return state["y"]
    if kind == "conv2d":
        k, pad = case["k"], case["pad"]
        for c in state["calls"]:
            A.alcs_spconv2d(c["w"], c["x"], c["y"], case["n"], c["ci"], c["h"], c["wd"], k, k, c["s"], pad, c["bias"], A.ALCS_RELU, stream)
        return [c["y"] for c in state["calls"]]
    if kind == "host":
        ws = state["ws"]
        A.alcs_spconv1x1_host(state["w"], state["x"], state["y"], case["n"], case["h"], case["w"], state["bias"], A.ALCS_RELU, ws,
                              ws.numel(), stream)
        return state["y"]
    r = A.alcs_project_bisection(state["u"], case["g"], state["tabs"], state["tau"], state["budget"], state["eps"], state["mask"],
                                 state["out"], stream)
    return {"mask": state["mask"], "u": state["out"], "n_keep": r["n_keep"], "kept_per_layer": np.array(r["kept_per_layer"])}


def _conv_work(nb, g, elt, y_elt, cout, x_elems, y_elems, q, bias=True, residual=False):
    """Kept weights times pixels; the packed weights, the inputs that are read, bias, residual and output once."""
    b = nb * (g * elt + 4) + x_elems * elt + y_elems * y_elt * (2 if residual else 1) + (4 * cout if bias else 0)
    return b, 2.0 * nb * g * q


def work(case):
    kind, by, fl = case["kind"], 0.0, 0.0
    if kind in ("layer", "host"):
        g, elt, s = case["g"], _ELT[case["dtype"]], case.get("stride", 1)
        q = case["n"] * _up(case["h"], s) * _up(case["w"], s)
        rows = _up(case["cout"], g)
        if case.get("rows") == "zipf":
            nb = rows * float((np.arange(1, case["cin"] + 1) * _zipf_pmf(case["cin"])).sum())
        else:
            nb = _kept(rows, case["cin"], case["sparsity"])
        by, fl = _conv_work(nb, g, elt, 4 if case.get("y_f32") else elt, case["cout"], q * case["cin"], q * case["cout"], q,
                            case.get("bias", True), case.get("residual", False))
        if kind == "host":      # what crosses the bus also passes through device memory once
            by += (q * case["cin"] + q * case["cout"]) * elt
    elif kind == "stack":
        table, g, elt = _net_layers(case), case["g"], _ELT[case["dtype"]]
        for (ci, co, s), sp in zip(table, _sparsities(case, len(table))):
            q = case["n"] * s * s
            b, f = _conv_work(_kept(_up(co, g), ci, sp), g, elt, elt, co, q * ci, q * co, q)
            by, fl = by + b, fl + f
    elif kind == "conv2d":
        k, pad, g = case["k"], case["pad"], case["g"]
        for ci, co, h, w, s in _conv_layers(case):
            q = case["n"] * ((h + 2 * pad - k) // s + 1) * ((w + 2 * pad - k) // s + 1)
            b, f = _conv_work(_kept(_up(co, g), ci * k * k, case["sparsity"]), g, 4, 4, co, case["n"] * ci * h * w, q * co, q)
            by, fl = by + b, fl + f
    else:
        for ci, co, _ in _net_layers(case):      # weights read, projected weights and one mask byte per group written
            by += 8.0 * ci * co + _up(co, case["g"]) * ci
            fl += 2.0 * ci * co
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    if case["kind"] == "project":
        return "exact"
    if case["kind"] == "conv2d" or case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}        # fp32 sums in another order
    if case.get("y_f32"):
        return {"rel": 1e-5, "max": 1e-4}        # exact products of 16-bit operands, fp32 sums, fp32 output
    return {"rel": 1e-3, "max": 4e-3} if case["dtype"] == "f16" else {"rel": 8e-3, "max": 3e-2}    # one rounding of the output
