"""GPU parity of the tcgen05 kernel for 16-bit operands (math_mode 4, producer_warps 8) against the oracle at the sizes where
its tiles, accumulators, copies and stores change."""
import numpy as np
import pytest

import oracle
from alcs_workloads import rng
from gpu_util import TOL, assert_parity, check_layer

pytestmark = pytest.mark.gpu
CFG = dict(math_mode=4, producer_warps=8)


def _case(seed, n, cin, cout, hw, g, density, dtype=np.float16):
    rows = (cout + g - 1) // g
    W = (rng.normal(seed, 1, cout * cin) * cin ** -0.5).reshape(cout, cin).astype(dtype)
    X = np.abs(rng.normal(seed, 2, n * cin * hw)).reshape(n, cin, hw).astype(dtype)
    M = (rng.uniform01(seed, 3, rows * cin) < density).astype(np.uint8).reshape(rows, cin)
    return W, M, X, (0.1 * rng.normal(seed, 4, cout)).astype(np.float32)


# n, cin, cout, h, wd, g, density: one pixel; ends of pixel tiles (31 .. 33, 255 .. 257 pixels); columns around a chunk and around an
# accumulator (63 .. 65, 255 .. 257); channels around a tile and around a warp's 32; copies of 16, 8 bytes and fetched rows, images that
# end inside a copy; column lists; more items than SMs, with one accumulator and with several
SHAPES = [(1, 16, 8, 1, 1, 8, 1.0), (1, 63, 127, 31, 1, 8, 0.4), (2, 64, 128, 4, 4, 8, 0.4), (1, 65, 129, 33, 1, 8, 0.4), (1, 255, 33, 255, 1, 1, 0.3),
          (1, 256, 31, 16, 16, 16, 0.3), (1, 257, 130, 257, 1, 8, 0.3), (3, 40, 72, 14, 14, 8, 0.3), (5, 100, 64, 7, 7, 8, 0.4), (4, 48, 40, 9, 6, 8, 0.4),
          (3, 520, 96, 17, 23, 8, 0.2), (7, 300, 64, 6, 6, 4, 0.02), (24, 64, 256, 28, 28, 8, 0.25), (30, 272, 260, 14, 14, 8, 0.25), (9, 16, 16, 56, 56, 8, 1.0)]


@pytest.mark.parametrize("n,cin,cout,h,wd,g,density", SHAPES)
def test_shapes(alcs, n, cin, cout, h, wd, g, density):
    W, M, X, b = _case(n + cin + cout, n, cin, cout, h * wd, g, density)
    for tiles in sorted({0, -(-cout // 16)}):
        check_layer(alcs, W, M, X, b, True, g, cfg=dict(CFG, row_groups=tiles), h=h, wd=wd)
    # fp32 output: the products are exact, so the fp32 tolerance holds
    Y = check_layer(alcs, W, M, X, None, False, g, cfg=CFG, h=h, wd=wd, y_f32=True)
    assert Y <= TOL["f32"]


def _device_call(alcs, W, M, X, b, g, h, wd, res, bf16, y_f32, x_off=0, y_off=0, cfg=CFG):
    """One residual call with X and Y starting `off` elements into their buffers; returns Y and what lies around it."""
    import torch
    dev = torch.device("cuda:0")
    tdt = torch.bfloat16 if bf16 else torch.float16
    Wt = torch.from_numpy(W.astype(np.float32)).to(tdt)
    p = alcs.alcs_pack(Wt.view(torch.int16).numpy().view(np.uint16), M, g, bf16=True) if bf16 else alcs.alcs_pack(Wt.numpy(), M, g)
    alcs.alcs_packed_upload(p, 0)
    n, cin, hw = X.shape
    xb = torch.zeros(X.size + x_off + 8, dtype=tdt, device=dev)
    xb[x_off:x_off + X.size] = torch.from_numpy(X.astype(np.float32)).to(dev).to(tdt).reshape(-1)
    ydt = torch.float32 if y_f32 else tdt
    size = n * W.shape[0] * hw
    yb = torch.full((size + y_off + 32,), 7.0, dtype=ydt, device=dev)
    rt = None if res is None else torch.from_numpy(res).to(dev).to(ydt).contiguous()
    flags = alcs.ALCS_RELU | (alcs.ALCS_Y_F32 if y_f32 else 0)
    alcs.alcs_spconv1x1_ex(p, xb[x_off:], yb[y_off:], n, h, wd, 1, torch.from_numpy(b).to(dev), rt, flags, torch.cuda.current_stream(), cfg)
    torch.cuda.synchronize()
    assert alcs.alcs_packed_status(p) == 0
    y = yb.float().cpu().numpy()
    assert (y[:y_off] == 7).all() and (y[y_off + size:] == 7).all(), "stored outside Y"
    x = xb[x_off:x_off + X.size].float().cpu().numpy().reshape(X.shape)
    return y[y_off:y_off + size].reshape(n, W.shape[0], hw), Wt.float().numpy(), x, None if rt is None else rt.float().cpu().numpy()


@pytest.mark.parametrize("n,cin,cout,h,wd", [(3, 64, 136, 7, 7), (2, 48, 40, 14, 14), (4, 272, 96, 8, 8), (2, 33, 260, 11, 13), (40, 40, 136, 16, 16)])
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("y_f32", [False, True])
@pytest.mark.parametrize("offsets", [(0, 0), (4, 2), (1, 1)])
def test_residual_types_and_alignments(alcs, n, cin, cout, h, wd, bf16, y_f32, offsets):
    """Residual, output types, and buffers that start anywhere.  One rounding of the output: 2^-11 of it in fp16, 2^-8 in bfloat16
    (half of the last place kept, doubled), beside the fp32 sum's tolerance."""
    g, hw = 8, h * wd
    W, M, X, b = _case(cin + cout, n, cin, cout, hw, g, 0.4, np.float32)
    res = rng.normal(9, 5, n * cout * hw).reshape(n, cout, hw).astype(np.float32)
    Y, Wr, Xr, Rr = _device_call(alcs, W, M, X, b, g, h, wd, res, bf16, y_f32, *offsets)
    Yref, A = oracle.conv1x1(Wr, M, Xr, b, False, g, want_scale=True)
    Yref, A = np.maximum(Yref + Rr, 0.0), A + np.abs(Rr)
    assert np.isfinite(Y).all()
    unit = 0.0 if y_f32 else 2.0 ** -8 if bf16 else 2.0 ** -11
    assert (np.abs(Y - Yref) <= TOL["f32"] * A + unit * np.abs(Yref)).all()


@pytest.mark.parametrize("x_off", [0, 1, 3, 7])
@pytest.mark.parametrize("n,hw", [(1, 49), (2, 63), (3, 131)])
def test_ends_of_x_in_slots_used_again(alcs, n, hw, x_off):
    """Words that reach beyond X are stored element by element, to slots that held other rows before: six chunks, sixteen channel
    tiles, and other values at the second call."""
    g, cin, cout = 8, 384, 256
    for seed in (3, 4):
        W, M, X, b = _case(seed, n, cin, cout, hw, g, 0.4, np.float32)
        Y, Wr, Xr, _ = _device_call(alcs, W, M, X, b, g, hw, 1, None, False, True, x_off, cfg=dict(CFG, row_groups=16))
        Yref, A = oracle.conv1x1(Wr, M, Xr, b, True, g, want_scale=True)
        assert (np.abs(Y - Yref) <= TOL["f32"] * A).all()


def test_rows_that_keep_nothing_and_skewed_rows(alcs):
    n, cin, cout, h, g = 6, 300, 256, 14, 8
    W, M, X, b = _case(5, n, cin, cout, h * h, g, 0.05)
    M[3::2] = 0
    M[0] = 1
    for tiles in (2, 8, 16):
        check_layer(alcs, W, M, X, b, True, g, cfg=dict(CFG, row_groups=tiles), h=h, wd=h)
    M[:] = 0
    Y = check_layer(alcs, W, M, X, b, True, g, cfg=CFG, h=h, wd=h)
    assert Y <= 2.0 ** -11


@pytest.mark.parametrize("h,cin", [(14, 64), (7, 300), (8, 272)])
def test_infinite_and_nan_inputs_touch_kept_blocks_alone(alcs, h, cin):
    n, cout, g = 3, 136, 8
    W, M, X, b = _case(31, n, cin, cout, h * h, g, 0.3)
    X[1, 5, 3] = np.inf
    X[2, 7, h * h - 1] = np.nan
    import torch
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    x, y = torch.from_numpy(X).cuda(), torch.empty(n, cout, h * h, dtype=torch.float16, device="cuda")
    alcs.alcs_spconv1x1(p, x, y, n, h, h, torch.from_numpy(b).cuda(), 0, torch.cuda.current_stream(), CFG)
    torch.cuda.synchronize()
    Y = y.float().cpu().numpy()
    kept = np.repeat(M, g, axis=0)[:cout].astype(bool)
    Xf = X.copy()
    Xf[1, 5, 3] = Xf[2, 7, h * h - 1] = 0
    Yref, A = oracle.conv1x1(W, M, Xf, b, False, g, want_scale=True)
    bad = np.zeros(Y.shape, bool)
    bad[1, kept[:, 5] & (W[:, 5] != 0), 3] = True
    bad[2, kept[:, 7], h * h - 1] = True
    assert not np.isfinite(Y[bad]).any()
    assert_parity(np.where(bad, 0, Y), np.where(bad, 0, Yref), A, "f16")


def _kernels(alcs, s, count):
    cfgs = [alcs.alcs_stack_layer_cfg(s, i) for i in range(count)]
    assert all(c["math_mode"] == 4 for c in cfgs)
    return [c["producer_warps"] for c in cfgs]


@pytest.mark.parametrize("sizes", [[(64, 96, 14), (272, 40, 8), (32, 160, 28)], [(48, 64, 16), (100, 64, 7), (64, 32, 14)]])
@pytest.mark.parametrize("kernels", [[8, 8, 8], [8, 4, 8], [4, 8, 8]])
@pytest.mark.parametrize("graph", [False, True])
def test_merged_stack(alcs, sizes, kernels, graph):
    """Layers of one launch, and layers of the two tensor-core kernels one behind the other."""
    import torch
    n, g = 6, 8
    layers, want = [], []
    for i, (cin, cout, h) in enumerate(sizes):
        W, M, X, b = _case(100 + i, n, cin, cout, h * h, g, 0.4)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
        alcs.alcs_spconv1x1_set_cfg(p, n, h, h, alcs.ALCS_RELU, dict(math_mode=4, producer_warps=kernels[i]))
        layers.append(dict(w=p, x=torch.from_numpy(X).cuda(), y=torch.full((n, cout, h * h), float("nan"), dtype=torch.float16, device="cuda"),
                           n=n, h=h, wd=h, bias=torch.from_numpy(b).cuda(), flags=alcs.ALCS_RELU))
        want.append(oracle.conv1x1(W, M, X, b, True, g, want_scale=True))
    s = alcs.alcs_stack_create(layers, alcs.ALCS_STACK_GRAPH if graph else 0)
    assert _kernels(alcs, s, 3) == kernels
    for _ in range(2):
        alcs.alcs_stack_run(s, torch.cuda.current_stream())
    torch.cuda.synchronize()
    for L, (Yref, A) in zip(layers, want):
        assert_parity(L["y"].cpu().numpy(), Yref, A, "f16")
        assert alcs.alcs_packed_status(L["w"]) == 0


def test_stack_that_runs_as_two_launches(alcs):
    """ResNet-50's pointwise layers at 224: the two of 7x7 images run on the other kernel, in a launch of their own."""
    import torch
    from alcs_workloads.layers import RESNET50_BOTTLENECK_PW
    n, g, gen = 32, 8, torch.Generator("cuda").manual_seed(5)
    layers, ws = [], []
    for i, (cin, cout, h) in enumerate(RESNET50_BOTTLENECK_PW):
        W, M, _, b = _case(200 + i, 1, cin, cout, 1, g, 0.25)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
        x = torch.randn(n, cin, h * h, generator=gen, device="cuda").abs_().half()
        layers.append(dict(w=p, x=x, y=torch.full((n, cout, h * h), float("nan"), dtype=torch.float16, device="cuda"), n=n, h=h, wd=h,
                           bias=torch.from_numpy(b).cuda(), flags=0))
        ws.append(torch.from_numpy(W.astype(np.float64) * np.repeat(M, g, axis=0)[:cout]).cuda())
    s = alcs.alcs_stack_create(layers, 0)
    assert _kernels(alcs, s, len(layers)) == [4 if h == 7 else 8 for _, _, h in RESNET50_BOTTLENECK_PW]
    alcs.alcs_stack_run(s, torch.cuda.current_stream())
    torch.cuda.synchronize()
    for L, W in zip(layers, ws):
        x, b = L["x"].double(), L["bias"].double()[:, None]
        Yref, A = W @ x + b, W.abs() @ x + b.abs()
        assert ((L["y"].double() - Yref).abs() <= TOL["f32"] * A + 2.0 ** -11 * Yref.abs() + 2.0 ** -25).all()


@pytest.mark.parametrize("bf16", [False, True])
def test_merged_launch_of_unlike_layers(alcs, bf16):
    """One launch of the kernel with a residual, fp32 output, an X that starts on an odd element and infinite and NaN inputs, in different
    layers: each keeps to itself."""
    import torch
    n, g, dt = 5, 8, torch.bfloat16 if bf16 else torch.float16
    kinds = ["plain", "residual", "y_f32", "odd start", "not finite", "y_f32 residual", "plain"]
    sizes = [(64, 96, 14), (272, 136, 8), (32, 160, 28), (100, 72, 10), (300, 136, 14), (64, 40, 12), (48, 64, 16)]
    layers, refs, st = [], [], torch.cuda.current_stream()
    for i, (kind, (cin, cout, h)) in enumerate(zip(kinds, sizes)):
        W, M, X, b = _case(300 + i, n, cin, cout, h * h, g, 0.4, np.float32)
        Wt = torch.from_numpy(W).to(dt)
        p = alcs.alcs_pack(Wt.view(torch.int16).numpy().view(np.uint16), M, g, bf16=True) if bf16 else alcs.alcs_pack(Wt.numpy(), M, g)
        alcs.alcs_packed_upload(p, 0)
        flags = alcs.ALCS_Y_F32 if "y_f32" in kind else 0
        alcs.alcs_spconv1x1_set_cfg(p, n, h, h, flags, CFG)
        off = 1 if kind == "odd start" else 0
        x = torch.zeros(X.size + 8, dtype=dt, device="cuda")[off:off + X.size].view(X.shape)
        x.copy_(torch.from_numpy(X))
        if kind == "not finite":
            x[1, 5, 3], x[2, 7, h * h - 1] = float("inf"), float("nan")
        ydt = torch.float32 if flags else dt
        res = torch.from_numpy(rng.normal(9, i, n * cout * h * h).astype(np.float32)).cuda().to(ydt).view(n, cout, h * h) if "residual" in kind else None
        layers.append(dict(w=p, x=x, y=torch.full((n, cout, h * h), 7.0, dtype=ydt, device="cuda"), n=n, h=h, wd=h, bias=torch.from_numpy(b).cuda(),
                           flags=flags, residual=res))
        refs.append((Wt.double().cuda() * torch.from_numpy(np.repeat(M, g, axis=0)[:cout]).cuda(), M))
    s = alcs.alcs_stack_create(layers, 0)
    assert _kernels(alcs, s, len(layers)) == [8] * len(layers)
    alcs.alcs_stack_run(s, st)
    torch.cuda.synchronize()
    for kind, L, (W, M) in zip(kinds, layers, refs):
        x, b, bad = L["x"].double(), L["bias"].double()[:, None], torch.zeros_like(L["y"], dtype=torch.bool)
        if kind == "not finite":
            kept = torch.from_numpy(np.repeat(M, g, axis=0)[:W.shape[0]]).cuda().bool()
            bad[1, :, 3], bad[2, :, -1] = kept[:, 5] & (W[:, 5] != 0), kept[:, 7]
            x = torch.where(x.isfinite(), x, torch.zeros_like(x))
        Yref, A = W @ x + b, W.abs() @ x.abs() + b.abs()
        if L["residual"] is not None:
            Yref, A = Yref + L["residual"].double(), A + L["residual"].double().abs()
        y, unit = L["y"].double(), 0.0 if L["y"].dtype == torch.float32 else 2.0 ** -8 if bf16 else 2.0 ** -11
        assert not y[bad].isfinite().any() and (bad.any() or kind != "not finite")
        assert ((y - Yref).abs() <= TOL["f32"] * A + unit * Yref.abs() + 2.0 ** -25)[~bad].all(), kind
        assert alcs.alcs_packed_status(L["w"]) == 0


@pytest.mark.parametrize("cin,h", [(64, 14), (300, 14), (64, 7), (300, 9)])
def test_configurations_say_what_runs(alcs, cin, h):
    """What plan() and a stack report names the kernel, its channel tiles and its pixels per tile, so that it can be fixed again."""
    n, cout, g = 4, 136, 8
    W, M, X, b = _case(cin + h, n, cin, cout, h * h, g, 0.4)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    most = (256 if h == 14 else 128) if cin == 64 else 128
    asked = [(0, 0), (4, 0), (8, 0), (8, -1)] + [(8, warps) for warps in (1, 2, 3, 4, 8, 100)]
    for producers, warps in asked:
        for tiles in (0, 2, 5):
            cfg = dict(math_mode=4, producer_warps=producers, pixels_per_lane=1, warps=warps, row_groups=tiles)
            alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, cfg)
            plan = alcs.alcs_spconv1x1_plan(p, n, h, h)
            assert plan["math_mode"] == 4 and (not tiles or plan["row_groups"] == tiles)
            assert plan["producer_warps"] == producers if producers else plan["producer_warps"] in (4, 8)
            if producers == 8:
                assert plan["warps"] in ([min(warps, most // 32)] if warps > 0 else range(1, most // 32 + 1))
            else:
                assert plan["warps"] == 0 or plan["producer_warps"] == 8
            assert plan["pixels_per_lane"] == 1
            alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, plan)
            assert alcs.alcs_spconv1x1_plan(p, n, h, h) == plan
            check_layer(alcs, W, M, X, b, False, g, cfg=plan, h=h, wd=h, packed=p)
    # in a stack, beside a layer on the other kernel
    import torch
    x, ys = torch.from_numpy(X).cuda(), [torch.empty(n, cout, h * h, dtype=torch.float16, device="cuda") for _ in range(3)]
    qs = [alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0) for _ in range(3)]
    want = [dict(math_mode=4, producer_warps=8, warps=2, row_groups=2), dict(math_mode=4, producer_warps=4, warps=0, row_groups=3),
            dict(math_mode=4, producer_warps=8, warps=1, row_groups=9)]
    for q, cfg in zip(qs, want):
        alcs.alcs_spconv1x1_set_cfg(q, n, h, h, 0, cfg)
    s = alcs.alcs_stack_create([dict(w=q, x=x, y=y, n=n, h=h, wd=h, bias=None, flags=0) for q, y in zip(qs, ys)], 0)
    for i, cfg in enumerate(want):
        got = alcs.alcs_stack_layer_cfg(s, i)
        assert {k: got[k] for k in cfg} == cfg
    alcs.alcs_stack_run(s, torch.cuda.current_stream())
    torch.cuda.synchronize()
    Yref, A = oracle.conv1x1(W, M, X, None, False, g, want_scale=True)
    for y in ys:
        assert_parity(y.cpu().numpy(), Yref, A, "f16")


def test_layers_of_one_kernel_take_any_producers(alcs):
    """fp32 and strided layers have one tcgen05 kernel: producer_warps says nothing there, as ever."""
    import torch
    W, M, X, b = _case(3, 2, 64, 72, 14 * 14, 8, 0.5, np.float32)
    for producers in (0, 4, 8):
        check_layer(alcs, W, M, X, b, True, 8, cfg=dict(math_mode=4, producer_warps=producers), h=14, wd=14)
    W, M, X, b = _case(4, 2, 64, 72, 16 * 16, 8, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 8), 0)
    x, y = torch.from_numpy(X).cuda(), torch.empty(2, 72, 64, dtype=torch.float16, device="cuda")
    ref = None
    for producers in (0, 4, 8):
        alcs.alcs_spconv1x1_ex(p, x, y, 2, 16, 16, 2, None, None, 0, torch.cuda.current_stream(), dict(math_mode=4, producer_warps=producers))
        torch.cuda.synchronize()
        ref = y.clone() if ref is None else ref
        assert torch.equal(y, ref)


@pytest.mark.parametrize("stack", [False, True])
def test_tuners_compare_the_two_kernels(alcs, stack):
    """X starts on an odd word here, which rows fetched as they are pay for (49 us and more where the other kernel takes 25; for an aligned X
    it is the slower one): only a tuner that times both kernels finds out."""
    import torch
    n, cin, cout, h, g = 38, 78, 1300, 20, 8
    W, M, X, b = _case(12, n, cin, cout, h * h, g, 0.25, np.float32)
    Wt, st = torch.from_numpy(W).to(torch.bfloat16), torch.cuda.current_stream()
    x = torch.zeros(X.size + 8, dtype=torch.bfloat16, device="cuda")[2:2 + X.size]
    x.copy_(torch.from_numpy(X).reshape(-1))
    Yref, A = oracle.conv1x1(Wt.float().numpy(), M, x.float().cpu().numpy().reshape(X.shape), None, False, g, want_scale=True)
    ps = [alcs.alcs_packed_upload(alcs.alcs_pack(Wt.view(torch.int16).numpy().view(np.uint16), M, g, bf16=True), 0) for _ in range(2 if stack else 1)]
    ys = [torch.empty(n, cout, h * h, dtype=torch.bfloat16, device="cuda") for _ in ps]
    if stack:
        for p in ps:
            alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, dict(math_mode=4, producer_warps=8))
        s = alcs.alcs_stack_create([dict(w=p, x=x, y=y, n=n, h=h, wd=h, bias=None, flags=0) for p, y in zip(ps, ys)], 0)
        alcs.alcs_stack_tune(s, 1, st)
        alcs.alcs_stack_run(s, st)
        assert all(alcs.alcs_stack_layer_cfg(s, i)["producer_warps"] == 4 for i in range(2))
    else:
        alcs.alcs_spconv1x1_tune(ps[0], x, ys[0], n, h, h, None, 0, st)
    torch.cuda.synchronize()
    for p, y in zip(ps, ys):
        cfg = alcs.alcs_spconv1x1_plan(p, n, h, h)
        assert (cfg["math_mode"], cfg["producer_warps"]) == (4, 4)
        assert (np.abs(y.float().cpu().numpy() - Yref) <= TOL["f32"] * A + 2.0 ** -8 * np.abs(Yref)).all()


def test_planner_knows_the_output_type(alcs):
    """fp32 output stores (and reads as a residual) twice the bytes: 22 -> 45 channels @32x32 with a residual, batch 85, took 29 us on the kernel that the
    estimate for 16-bit output chose, 13 us before."""
    import torch
    n, cin, cout, h, g = 85, 22, 45, 32, 8
    W, M, X, b = _case(6, n, cin, cout, h * h, g, 0.165)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    x, bd, chosen = torch.from_numpy(X).cuda(), torch.from_numpy(b).cuda(), []
    for dt, flags in ((torch.float16, 0), (torch.float32, alcs.ALCS_Y_F32)):
        y, r = torch.empty(n, cout, h * h, dtype=dt, device="cuda"), torch.zeros(n, cout, h * h, dtype=dt, device="cuda")
        s = alcs.alcs_stack_create([dict(w=p, x=x, y=y, n=n, h=h, wd=h, bias=bd, flags=flags, residual=r)], 0)
        alcs.alcs_stack_run(s, torch.cuda.current_stream())
        torch.cuda.synchronize()
        Yref, A = oracle.conv1x1(W, M, X, b, False, g, want_scale=True)
        assert_parity(y.cpu().numpy(), Yref, A, "f16")
        cfg = alcs.alcs_stack_layer_cfg(s, 0)
        chosen.append(cfg["math_mode"] == 4 and cfg["producer_warps"] == 8)
    assert chosen == [True, False]


@pytest.mark.parametrize("n,cin,cout,h,w,density", [(31, 173, 247, 11, 13, 0.335), (3, 145, 578, 21, 21, 0.426), (16, 128, 256, 28, 28, 0.3), (8, 256, 96, 14, 14, 0.4),
                                                    (9, 64, 80, 7, 7, 0.4)])
def test_planned_tiles_are_the_best_of_their_kernel(alcs, n, cin, cout, h, w, density):
    """The width of the channel tiles follows from the estimate of the kernel that runs (217 images of 204 -> 115 channels @7x7 with a
    residual: 27 us with the 48 channels that suit the other kernel, 17 with 115)."""
    W, M, X, b = _case(8, n, cin, cout, h * w, 8, density)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 8), 0)
    plan = alcs.alcs_spconv1x1_plan(p, n, h, w)
    if plan["math_mode"] == 4:
        alcs.alcs_spconv1x1_set_cfg(p, n, h, w, 0, dict(math_mode=4, producer_warps=plan["producer_warps"]))
        assert alcs.alcs_spconv1x1_plan(p, n, h, w) == plan
    check_layer(alcs, W, M, X, b, True, 8, h=h, wd=w)


def test_inputs_that_start_on_odd_words(alcs):
    """A layer planned for rows copied as they are, whose X does not start where such copies can: 38 images of 78 -> 1300 channels @20x20 took
    153 us with 32 pixels per tile on the kernel that then picks rows apart, 49 with 128, 25 on the other one."""
    import torch
    n, cin, cout, h, g = 38, 78, 1300, 20, 8
    W, M, X, b = _case(12, n, cin, cout, h * h, g, 0.25)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    st, bd = torch.cuda.current_stream(), torch.from_numpy(b).cuda()
    x = torch.zeros(X.size + 8, dtype=torch.float16, device="cuda")[2:2 + X.size]
    x.copy_(torch.from_numpy(X).reshape(-1))
    y = torch.empty(n, cout, h * h, dtype=torch.float16, device="cuda")
    Yref, A = oracle.conv1x1(W, M, X, b, False, g, want_scale=True)
    assert alcs.alcs_spconv1x1_plan(p, n, h, h)["producer_warps"] == 8
    took = {}
    for cfg in (None, dict(CFG, warps=8), dict(CFG, warps=4), dict(CFG, warps=1), dict(math_mode=4, producer_warps=4)):
        for _ in range(3):
            y.fill_(float("nan"))
            alcs.alcs_spconv1x1(p, x, y, n, h, h, bd, 0, st, cfg)
        best = []
        for _ in range(5):
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                alcs.alcs_spconv1x1(p, x, y, n, h, h, bd, 0, st, cfg)
            e.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(e))
        took[tuple(cfg.values()) if cfg else None] = min(best)
        assert_parity(y.cpu().numpy(), Yref, A, "f16")
    times = list(took.values())
    assert times[1] < 1.5 * times[2] < 1.5 * times[3] and times[0] < 1.3 * times[4], took
    s = alcs.alcs_stack_create([dict(w=p, x=x, y=y, n=n, h=h, wd=h, bias=bd, flags=0)], 0)
    assert alcs.alcs_stack_layer_cfg(s, 0)["producer_warps"] == 4
    # without allocation, and in a captured graph
    y.fill_(float("nan"))
    alcs.alcs_spconv1x1_noalloc(p, x, y, n, h, h, bd, 0, st)
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), Yref, A, "f16")


def test_more_than_2_to_the_30_elements(alcs):
    """Byte offsets of rows picked apart pass 2^31: the last images of 1.18e9 elements, against the same images by themselves."""
    import torch
    n, cin, cout, hw, g = 18000, 16, 8, 4097, 8
    assert n * cin * hw > 2 ** 30
    W, M, _, b = _case(2, 1, cin, cout, 8, g, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    st, bd = torch.cuda.current_stream(), torch.from_numpy(b).cuda()
    x = torch.empty(n, cin, hw, dtype=torch.float16, device="cuda").uniform_(0, 1, generator=torch.Generator("cuda").manual_seed(1))
    y = torch.empty(n, cout, hw, dtype=torch.float16, device="cuda")
    alcs.alcs_spconv1x1(p, x, y, n, hw, 1, bd, 0, st, CFG)
    for first in (0, n // 2, n - 3):
        few = torch.empty(3, cout, hw, dtype=torch.float16, device="cuda")
        alcs.alcs_spconv1x1(p, x[first:first + 3].clone(), few, 3, hw, 1, bd, 0, st, CFG)
        torch.cuda.synchronize()
        assert torch.equal(y[first:first + 3], few)
    Yref, A = oracle.conv1x1(W, M, x[-3:].cpu().numpy(), b, False, g, want_scale=True)
    assert_parity(few.cpu().numpy(), Yref, A, "f16")
    assert alcs.alcs_packed_status(p) == 0
