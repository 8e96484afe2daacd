"""Which kernel a call is given, and what it does there: calls at the edge of what the tcgen05 kernel takes must run on
another kernel (or be refused), and give what the oracle gives."""
import numpy as np
import pytest

import oracle
from alcs_workloads import rng
from gpu_util import TOL, assert_parity, run_gpu

pytestmark = pytest.mark.gpu


def _case(seed, n, cin, cout, hw, g, density, dtype=np.float32):
    rows = (cout + g - 1) // g
    W = (rng.normal(seed, 1, cout * cin) * cin ** -0.5).reshape(cout, cin).astype(dtype)
    X = rng.normal(seed, 2, n * cin * hw).reshape(n, cin, hw).astype(dtype)
    M = (rng.uniform01(seed, 3, rows * cin) < density).astype(np.uint8).reshape(rows, cin)
    return W, M, X, (0.1 * rng.normal(seed, 4, cout)).astype(np.float32)


# n, cin, cout, h, wd, stride: rows of 26, 14 and 18 bytes; the first is large enough for the tensor cores to be the
# planner's first choice where they can be had
@pytest.mark.parametrize("n,cin,cout,h,wd,stride", [(64, 1024, 512, 13, 13, 2), (16, 512, 512, 7, 7, 2), (9, 300, 260, 11, 9, 3)])
@pytest.mark.parametrize("bf16", [False, True])
def test_strided_rows_that_cannot_be_copied_by_words(alcs, n, cin, cout, h, wd, stride, bf16):
    """16-bit rows of odd length: no tcgen05 plan, neither by default nor from a stride-1 call of the same output size."""
    import torch
    g = 8
    W, M, X, b = _case(n + cin, n, cin, cout, h * wd, g, 0.5, np.float32 if bf16 else np.float16)
    if bf16:
        wb, xb = rng.to_bf16_bits(W), rng.to_bf16_bits(X)
        W, X = oracle.bf16_decode(wb), oracle.bf16_decode(xb)
        p = alcs.alcs_pack(wb, M, g, bf16=True)
        xd = torch.from_numpy(xb.view(np.int16)).cuda().view(torch.bfloat16)
    else:
        p = alcs.alcs_pack(W, M, g)
        xd = torch.from_numpy(X).cuda()
    p = alcs.alcs_packed_upload(p, 0)
    st, oh, ow = torch.cuda.current_stream(), -(-h // stride), -(-wd // stride)
    xs = torch.zeros((n, cin, oh * ow), dtype=xd.dtype, device="cuda")
    res = torch.zeros((n, cout, oh * ow), device="cuda")
    y = torch.full((n, cout, oh * ow), float("nan"), device="cuda")
    alcs.alcs_spconv1x1_ex(p, xs, y, n, oh, ow, 1, None, res, alcs.ALCS_Y_F32, st)
    y.fill_(float("nan"))
    alcs.alcs_spconv1x1_ex(p, xd, y, n, h, wd, stride, torch.from_numpy(b).cuda(), None, alcs.ALCS_Y_F32, st)
    with pytest.raises(alcs.AlcsError) as e:
        alcs.alcs_spconv1x1_ex(p, xd, y, n, h, wd, stride, None, None, alcs.ALCS_Y_F32, st, dict(math_mode=4))
    assert e.value.status == alcs.ALCS_ERR_UNSUPPORTED
    torch.cuda.synchronize()
    Yref, A = oracle.conv1x1_ex(W, M, X.reshape(n, cin, h, wd), b, None, False, g, stride, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f32")      # exact 16-bit products, fp32 sums and output
    assert alcs.alcs_packed_status(p) == 0


def test_strided_input_beyond_32_bit_offsets(alcs):
    """2.2e9 input elements: the plan cached for a stride-1 call of the same output size must not be taken."""
    import torch
    n, cin, cout, h, g, s = 688, 256, 16, 112, 8, 2
    W, M, _, _ = _case(3, 1, cin, cout, 1, g, 0.5, np.float16)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    st, o = torch.cuda.current_stream(), h // s
    small = torch.ones((n, cin, o * o), dtype=torch.float16, device="cuda")
    y = torch.empty((n, cout, o * o), dtype=torch.float16, device="cuda")
    alcs.alcs_spconv1x1_ex(p, small, y, n, o, o, 1, None, torch.zeros_like(y), 0, st)
    torch.cuda.synchronize()
    del small
    x = torch.empty((n, cin, h * h), dtype=torch.float16, device="cuda").normal_()
    assert x.numel() > 2 ** 31
    alcs.alcs_spconv1x1_ex(p, x, y, n, h, h, s, None, None, 0, st)
    torch.cuda.synchronize()
    for i in (0, n // 2, n - 1):
        Yref, A = oracle.conv1x1_ex(W, M, x[i:i + 1].cpu().numpy().reshape(1, cin, h, h), None, None, False, g, s, want_scale=True)
        assert_parity(y[i:i + 1].cpu().numpy(), Yref, A, "f16")
    assert alcs.alcs_packed_status(p) == 0


def test_long_predecessor_does_not_exhaust_the_waits_of_its_successor(alcs):
    """One pixel tile of many columns keeps one SM busy for milliseconds while the next launch, whose thread blocks
    start on the idle SMs, has nothing to multiply yet; several in a row."""
    import torch
    cin, g = 1 << 18, 16
    p = alcs.alcs_packed_upload(alcs.alcs_pack(np.ones((16, cin), np.float32), np.ones((1, cin), np.uint8), g), 0)
    x, y = torch.ones((1, cin, 16), device="cuda"), torch.empty((1, 16, 16), device="cuda")
    W, M, X, _ = _case(8, 40, 64, 32, 196, 4, 0.5)
    q = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
    xs, ys = torch.from_numpy(X).cuda(), torch.empty((40, 32, 196), device="cuda")
    st = torch.cuda.current_stream()
    for _ in range(3):
        for _ in range(4):
            alcs.alcs_spconv1x1(p, x, y, 1, 4, 4, None, 0, st, dict(math_mode=4))
        ys.fill_(float("nan"))
        alcs.alcs_spconv1x1(p, x, y, 1, 4, 4, None, 0, st, dict(math_mode=4))
        alcs.alcs_spconv1x1(q, xs, ys, 40, 14, 14, None, 0, st, dict(math_mode=4))
    torch.cuda.synchronize()
    assert (y.cpu().numpy() == cin).all()
    Yref, A = oracle.conv1x1(W, M, X, None, False, 4, want_scale=True)
    assert_parity(ys.cpu().numpy(), Yref, A, "f32")
    assert alcs.alcs_packed_status(p) == 0 and alcs.alcs_packed_status(q) == 0


def _with_specials(X, seed, share=1e-3):
    """X with infinities of both signs and NaNs among its values: scattered, and one pixel of nothing else."""
    X = X.copy()
    flat = X.reshape(-1)
    u = rng.uniform01(seed, 9, flat.size)
    for k, v in enumerate((np.inf, -np.inf, np.nan)):
        flat[(u >= k * share) & (u < (k + 1) * share)] = v
    X[-1, :, -1] = np.inf
    return X


def _kept_blocks_reference(W, M, X, b, g, residual=None):
    """Sums over the kept blocks alone, [n, cout, pixels] in float64, and the scale of their finite part.  (The oracle is
    dense: there 0 times an infinity is NaN for dropped blocks, too.)  W [cout, columns], X [n, columns, pixels]."""
    cout = W.shape[0]
    keep = np.repeat(M != 0, g, axis=0)[:cout]
    Wm, X = np.where(keep, W, 0).astype(np.float64), X.astype(np.float64)
    finite = np.where(np.isfinite(X), X, 0.0)
    base = 0.0 if b is None else b[None, :, None].astype(np.float64)
    Y, A = np.matmul(Wm, finite) + base, np.matmul(np.abs(Wm), np.abs(finite)) + np.abs(base)
    if residual is not None:
        Y, A = Y + residual, A + np.abs(residual)
    hits = lambda w, x: np.matmul(w.astype(np.float64), x.astype(np.float64)) > 0
    up, down, zero = keep & (Wm > 0), keep & (Wm < 0), keep & (Wm == 0)
    pos = hits(up, X == np.inf) | hits(down, X == -np.inf)
    neg = hits(up, X == -np.inf) | hits(down, X == np.inf)
    nan = hits(keep, np.isnan(X)) | hits(zero, np.isinf(X)) | (pos & neg)
    Y[pos], Y[neg], Y[nan] = np.inf, -np.inf, np.nan
    return Y, A


def _assert_special(Y, Yref, A, kind, relu=False):
    """Finite where the kept blocks meet finite values only, else the same infinity, or NaN (which a ReLU makes 0)."""
    Y = Y.reshape(Yref.shape).astype(np.float64)
    nan, inf = np.isnan(Yref), np.isinf(Yref)
    if relu:
        Yref = np.where(nan, Yref, np.maximum(Yref, 0.0))
    assert (Y[nan] == 0).all() if relu else np.isnan(Y[nan]).all()
    assert np.array_equal(Y[inf], Yref[inf])
    ok = ~nan & ~inf
    assert (np.abs(Y[ok] - Yref[ok]) <= TOL[kind] * A[ok]).all()
    assert not ok.all() and ok.any()


# n, cin, cout, h, wd, g, density: word and element copies, whole images, sorted rows with column lists, several chunks
@pytest.mark.parametrize("n,cin,cout,h,wd,g,density", [(3, 100, 150, 14, 14, 4, 0.3), (5, 65, 40, 9, 9, 2, 0.4), (7, 64, 260, 7, 7, 8, 0.3),
                                                      (2, 300, 128, 16, 16, 4, 0.0), (40, 200, 64, 12, 12, 1, 0.2)])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("relu", [False, True])
def test_infinite_and_nan_inputs_touch_kept_blocks_alone(alcs, n, cin, cout, h, wd, g, density, dtype, relu):
    W, M, X, b = _case(n + cin + cout, n, cin, cout, h * wd, g, density, dtype)
    if density == 0.0:
        M = (np.arange(cin)[None, :] < 1 + (np.arange(M.shape[0])[:, None] * 7) ** 2 % cin).astype(np.uint8)
    X = _with_specials(X, n)
    Yref, A = _kept_blocks_reference(W, M, X, b, g)
    for y_f32 in {False, dtype == np.float16}:
        Y = run_gpu(alcs, W, M, X, b, relu, g, cfg=dict(math_mode=4), y_f32=y_f32, h=h, wd=wd)
        _assert_special(Y, Yref, A, "f32" if dtype == np.float32 else "f16", relu)


@pytest.mark.parametrize("stride,dtype", [(1, np.float32), (2, np.float32), (2, np.float16)])
def test_infinite_and_nan_inputs_with_stride_and_residual(alcs, stride, dtype):
    import torch
    n, cin, cout, h, wd, g = 3, 72, 96, 12, 16, 8
    W, M, X, b = _case(stride, n, cin, cout, h * wd, g, 0.4, dtype)
    X = _with_specials(X, 5)
    oh, ow = -(-h // stride), -(-wd // stride)
    R = rng.normal(6, 5, n * cout * oh * ow).reshape(n, cout, oh * ow).astype(dtype)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    y = torch.zeros((n, cout, oh * ow), dtype=torch.float32 if dtype == np.float32 else torch.float16, device="cuda")
    alcs.alcs_spconv1x1_ex(p, torch.from_numpy(X).cuda(), y, n, h, wd, stride, torch.from_numpy(b).cuda(), torch.from_numpy(R).cuda(), 0,
                           torch.cuda.current_stream(), dict(math_mode=4))
    torch.cuda.synchronize()
    Xs = X.reshape(n, cin, h, wd)[:, :, ::stride, ::stride].reshape(n, cin, oh * ow)
    _assert_special(y.cpu().numpy(), *_kept_blocks_reference(W, M, Xs, b, g, R), "f32" if dtype == np.float32 else "f16")


@pytest.mark.parametrize("n,cin,cout,h,w,k,stride,pad", [(1, 200, 200, 7, 7, 3, 1, 1), (30, 40, 130, 14, 14, 3, 2, 1), (20, 65, 140, 9, 8, 3, 1, 0)])
def test_infinite_and_nan_inputs_of_a_kxk_layer(alcs, n, cin, cout, h, w, k, stride, pad):
    """(The first is small enough for its columns to be split; dense enough for the tensor cores.)"""
    import torch
    g = 1
    W, M, _, b = _case(n + cin, n, cin * k * k, cout, 1, g, 0.8)
    X = _with_specials(rng.normal(n + cin, 2, n * cin * h * w).reshape(n, cin, h * w).astype(np.float32), 7, 3e-4).reshape(n, cin, h, w)
    oh, ow = (h + 2 * pad - k) // stride + 1, (w + 2 * pad - k) // stride + 1
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    y = torch.zeros((n, cout, oh, ow), device="cuda")
    alcs.alcs_spconv2d(p, torch.from_numpy(X).cuda(), y, n, cin, h, w, k, k, stride, pad, torch.from_numpy(b).cuda(), 0, torch.cuda.current_stream())
    torch.cuda.synchronize()
    columns = torch.nn.functional.unfold(torch.from_numpy(X), k, padding=pad, stride=stride).numpy()
    _assert_special(y.cpu().numpy(), *_kept_blocks_reference(W, M, columns, b, g), "f32")


def test_infinite_inputs_of_one_layer_of_a_merged_stack(alcs):
    import torch
    layers, keep = [], []
    for i, (n, cin, cout, h) in enumerate([(2, 64, 96, 14), (3, 80, 48, 7), (2, 32, 160, 28)]):
        W, M, X, b = _case(60 + i, n, cin, cout, h * h, 4, 0.3)
        if i == 1:
            X = _with_specials(X, 3)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
        alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, dict(math_mode=4))
        layers.append(dict(w=p, x=torch.from_numpy(X).cuda(), y=torch.zeros((n, cout, h * h), device="cuda"), n=n, h=h, wd=h,
                           bias=torch.from_numpy(b).cuda(), flags=0))
        keep.append((X, oracle.conv1x1(W, M, X, b, False, 4, want_scale=True) if i != 1 else _kept_blocks_reference(W, M, X, b, 4)))
    st = alcs.alcs_stack_create(layers, 0)
    for _ in range(2):
        alcs.alcs_stack_run(st, torch.cuda.current_stream())
    torch.cuda.synchronize()
    for L, (X, (Yref, A)) in zip(layers, keep):
        (assert_parity if np.isfinite(X).all() else _assert_special)(L["y"].cpu().numpy(), Yref, A, "f32")
    alcs.alcs_stack_destroy(st)


def test_fp32_weights_that_are_not_finite(alcs):
    """An infinite weight has no bfloat16 parts that add up to it: such a matrix stays on the other kernels."""
    import torch
    n, cin, cout, h, g = 40, 96, 128, 14, 4
    W, M, X, b = _case(4, n, cin, cout, h * h, g, 0.5)
    X = np.abs(X) + np.float32(0.1)
    M[:, 0] = 1
    W[5, 0], W[70, 0], W[71, 0] = np.inf, -np.inf, np.nan
    M[3, 1] = 0
    W[12, 1] = np.nan                       # a dropped block's value is not kept
    p = alcs.alcs_packed_deserialize(alcs.alcs_packed_serialize(alcs.alcs_pack(W, M, g)))
    p = alcs.alcs_packed_upload(p, 0)
    st, xd, bd = torch.cuda.current_stream(), torch.from_numpy(X).cuda(), torch.from_numpy(b).cuda()
    y = [torch.full((n, cout, h * h), 7.0, device="cuda") for _ in range(3)]
    alcs.alcs_spconv1x1(p, xd, y[0], n, h, h, bd, 0, st)
    stack = alcs.alcs_stack_create([dict(w=p, x=xd, y=y[k], n=n, h=h, wd=h, bias=bd, flags=0) for k in (1, 2)], 0)
    alcs.alcs_stack_run(stack, st)
    with pytest.raises(alcs.AlcsError) as e:
        alcs.alcs_spconv1x1(p, xd, y[0], n, h, h, bd, 0, st, dict(math_mode=4))
    assert e.value.status == alcs.ALCS_ERR_UNSUPPORTED
    y2 = torch.full((n, cout, h, h), 7.0, device="cuda")
    alcs.alcs_spconv2d(p, xd, y2, n, cin, h, h, 1, 1, 1, 0, bd, 0, st)
    torch.cuda.synchronize()
    other = np.setdiff1d(np.arange(cout), (5, 70, 71))
    Wf = np.where(np.isfinite(W), W, 0).astype(np.float32)
    Yref, A = oracle.conv1x1(Wf, M, X, b, False, g, want_scale=True)
    for t in y + [y2]:
        Y = t.cpu().numpy().reshape(n, cout, h * h)
        assert (Y[:, 5] == np.inf).all() and (Y[:, 70] == -np.inf).all() and np.isnan(Y[:, 71]).all()
        assert_parity(Y[:, other], Yref[:, other], A[:, other], "f32")
    alcs.alcs_stack_destroy(stack)


def test_noalloc_after_stack_create(alcs):
    """Creating a stack makes its shapes usable without allocation, also where the layers were merged into one launch
    with other tiles than a layer by itself would get."""
    import torch
    layers, keep = [], []
    for i, (cin, cout, h) in enumerate([(64, 128, 56), (128, 256, 28), (512, 512, 14), (512, 512, 14), (1024, 1024, 7), (256, 256, 28)]):
        W, M, X, b = _case(80 + i, 1, cin, cout, h * h, 4, 0.2)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
        layers.append(dict(w=p, x=torch.from_numpy(X).cuda(), y=torch.empty((1, cout, h * h), device="cuda"), n=1, h=h, wd=h,
                           bias=torch.from_numpy(b).cuda(), flags=alcs.ALCS_RELU))
        keep.append(oracle.conv1x1(W, M, X, b, True, 4, want_scale=True))
    st = alcs.alcs_stack_create(layers, 0)
    for L, (Yref, A) in zip(layers, keep):
        y = torch.full_like(L["y"], float("nan"))
        alcs.alcs_spconv1x1_noalloc(L["w"], L["x"], y, 1, L["h"], L["wd"], L["bias"], L["flags"], torch.cuda.current_stream())
        torch.cuda.synchronize()
        assert_parity(y.cpu().numpy(), Yref, A, "f32")
    alcs.alcs_stack_destroy(st)


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("n,cin,cout,h,wd,stride", [(5, 64, 40, 7, 7, 1), (3, 80, 48, 14, 14, 1), (2, 64, 48, 12, 16, 2), (3, 100, 260, 9, 8, 2)])
def test_inputs_that_start_anywhere_take_what_the_first_call_prepared(alcs, n, cin, cout, h, wd, stride, dtype):
    """After one call for a shape, an X that starts on any element allocates nothing: it can be captured."""
    import torch
    g = 8
    W, M, X, b = _case(n + cin, n, cin, cout, h * wd, g, 0.4, dtype)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    oh, ow = -(-h // stride), -(-wd // stride)
    room = torch.empty(X.size + 8, dtype=torch.from_numpy(X).dtype, device="cuda")
    y = torch.empty((n, cout, oh * ow), dtype=room.dtype, device="cuda")
    bd = torch.from_numpy(b).cuda()
    side = torch.cuda.Stream()
    call = lambda x: alcs.alcs_spconv1x1_ex(p, x, y, n, h, wd, stride, bd, None, alcs.ALCS_RELU, side, dict(math_mode=4))
    Yref, A = oracle.conv1x1_ex(W, M, X.reshape(n, cin, h, wd), b, None, True, g, stride, want_scale=True)
    for at in range(8):
        x = room[at:at + X.size]
        x.copy_(torch.from_numpy(X).reshape(-1))
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        if at == 0:
            call(x)
        else:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=side):
                call(x)
            graph.replay()
        torch.cuda.synchronize()
        assert_parity(y.cpu().numpy(), Yref, A, "f32" if dtype == np.float32 else "f16")
        if stride == 1:
            alcs.alcs_spconv1x1_set_cfg(p, n, h, wd, alcs.ALCS_RELU, dict(math_mode=4))
            y.fill_(float("nan"))
            alcs.alcs_spconv1x1_noalloc(p, x, y, n, h, wd, bd, alcs.ALCS_RELU, torch.cuda.current_stream())
            torch.cuda.synchronize()
            assert_parity(y.cpu().numpy(), Yref, A, "f32" if dtype == np.float32 else "f16")
    assert alcs.alcs_packed_status(p) == 0


def test_host_call_in_pieces_keeps_the_configuration_of_its_shape(alcs):
    """The kernels differ in the order of their sums, so equal bits show that the same one ran."""
    import torch
    n, cin, cout, h, g = 32, 128, 128, 14, 4
    W, M, X, _ = _case(2, n, cin, cout, h * h, g, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    size = alcs.alcs_spconv1x1_host_workspace(p, n, h, h, 0)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    xh, yh = torch.from_numpy(X).pin_memory(), torch.empty((n, cout, h * h)).pin_memory()
    st, xd = torch.cuda.current_stream(), torch.from_numpy(X).cuda()
    results = []
    for cfg in (dict(math_mode=1), dict(math_mode=4, row_groups=2), dict(math_mode=3, pixels_per_lane=2, warps=4)):
        alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, cfg)
        alcs.alcs_spconv1x1_host(p, xh, yh, n, h, h, None, 0, ws, size, st)
        y = torch.empty((n, cout, h * h), device="cuda")
        alcs.alcs_spconv1x1(p, xd, y, n, h, h, None, 0, st)
        torch.cuda.synchronize()
        assert torch.equal(y.cpu(), yh)          # a pixel's sum does not depend on the images beside it
        results.append(yh.numpy().copy())
    assert not np.array_equal(results[0], results[1])         # (the kernels do differ in their rounding)


def _host_case(alcs, n=24, cin=128, cout=160, h=14):
    import torch
    W, M, X, b = _case(n, n, cin, cout, h * h, 4, 0.3)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
    size = alcs.alcs_spconv1x1_host_workspace(p, n, h, h, 0)
    call = lambda x, y, ws, st: alcs.alcs_spconv1x1_host(p, x, y, n, h, h, None, 0, ws, size, st)
    make = lambda: (torch.from_numpy(X).pin_memory(), torch.full((n, cout, h * h), float("nan")).pin_memory(),
                    torch.empty(size, dtype=torch.uint8, device="cuda"))
    return call, make, oracle.conv1x1(W, M, X, None, False, 4, want_scale=True)


def test_host_calls_do_not_wait_for_another_stream(alcs):
    """A call must end although a call on another stream, enqueued before it, cannot start yet.  (Few streams: more
    than the device has queues would wait for one another whatever the library does.)  Then more streams at once than
    the library keeps copy streams for."""
    import torch
    call, make, (Yref, A) = _host_case(alcs)
    free, slow, blocked = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.Stream()
    mine, theirs, gate = make(), make(), torch.cuda.Event()
    call(*mine, free)
    torch.cuda.synchronize()
    mine[1].fill_(float("nan"))
    with torch.cuda.stream(slow):
        torch.cuda._sleep(1_000_000_000)        # (half a second, on the device)
        gate.record(slow)
    blocked.wait_event(gate)
    call(*theirs, blocked)
    call(*mine, free)
    free.synchronize()
    assert not gate.query()
    torch.cuda.synchronize()
    many = [(torch.cuda.Stream(), make()) for _ in range(10)]
    with torch.cuda.stream(slow):
        torch.cuda._sleep(100_000_000)
        gate.record(slow)
    for s, b in many:
        s.wait_event(gate)
        call(*b, s)
    torch.cuda.synchronize()
    for b in [mine, theirs] + [b for _, b in many]:
        assert_parity(b[1].numpy(), Yref, A, "f32")


def test_host_call_under_capture(alcs):
    """The copies of a captured call are its graph's own: another stream's call during the capture is not drawn in."""
    import torch
    call, make, (Yref, A) = _host_case(alcs)
    a, b, side, other = make(), make(), torch.cuda.Stream(), torch.cuda.Stream()
    call(*a, side)
    call(*b, other)
    torch.cuda.synchronize()
    a[1].fill_(float("nan"))
    b[1].fill_(float("nan"))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="relaxed"):
        call(*a, side)
        call(*b, other)
    other.synchronize()
    assert_parity(b[1].numpy(), Yref, A, "f32")
    assert not np.isfinite(a[1].numpy()).any()
    graph.replay()
    torch.cuda.synchronize()
    assert_parity(a[1].numpy(), Yref, A, "f32")


def test_host_call_on_pageable_memory(alcs):
    """Pageable buffers, and a mix of both kinds, take the call in one piece."""
    import torch
    call, make, (Yref, A) = _host_case(alcs)
    x, y, ws = make()
    xp, yp = x.clone(), torch.empty(y.shape)
    assert not xp.is_pinned() and not yp.is_pinned()
    st = torch.cuda.current_stream()
    for a, b in ((x, y), (xp, yp), (x, yp), (xp, y)):
        b.fill_(float("nan"))
        call(a, b, ws, st)
        torch.cuda.synchronize()
        assert_parity(b.numpy(), Yref, A, "f32")


def test_graph_stack_survives_a_tuning_call_that_finds_no_memory(alcs):
    """alcs_stack_tune asks for scratch for every plan it may try; without the memory the stack runs on as before."""
    import torch
    W, M, X, b = _case(1, 40, 64, 48, 49, 4, 0.4)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
    alcs.alcs_spconv1x1_set_cfg(p, 40, 7, 7, 0, dict(math_mode=1))          # repacks its 7x7 images into the stack's scratch
    n, cin = 65536, 256
    V, N, _, _ = _case(2, 1, cin, 16, 49, 4, 0.5)
    big = alcs.alcs_packed_upload(alcs.alcs_pack(V, N, 4), 0)
    alcs.alcs_spconv1x1_set_cfg(big, n, 7, 7, 0, dict(math_mode=4))         # 3.3 GB of input, 4.3 GB of scratch for other plans
    y = torch.empty((40, 48, 49), device="cuda")
    layers = [dict(w=p, x=torch.from_numpy(X).cuda(), y=y, n=40, h=7, wd=7, bias=None, flags=0),
              dict(w=big, x=torch.zeros((n, cin, 49), device="cuda"), y=torch.empty((n, 16, 49), device="cuda"), n=n, h=7, wd=7, bias=None, flags=0)]
    st, s = alcs.alcs_stack_create(layers, alcs.ALCS_STACK_GRAPH), torch.cuda.Stream()
    alcs.alcs_stack_run(st, s)
    s.synchronize()
    Yref, A = oracle.conv1x1(W, M, X, None, False, 4, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f32")
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    with pytest.raises(alcs.AlcsError) as e:
        alcs.alcs_stack_tune(st, 1, s)
    assert e.value.status == alcs.ALCS_ERR_ALLOC
    del hog
    torch.cuda.empty_cache()
    other = torch.full((1 << 20,), 7.0, device="cuda")          # what a freed block would be given to
    for _ in range(2):
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        alcs.alcs_stack_run(st, s)
        s.synchronize()
        assert_parity(y.cpu().numpy(), Yref, A, "f32")
    assert (other == 7.0).all()
    alcs.alcs_stack_destroy(st)


def test_merged_layers_do_not_read_a_bias_that_another_one_writes(alcs):
    import torch
    n, cin, cout, h = 2, 64, 64, 14
    W, M, X, b = _case(9, n, cin, cout, h * h, 4, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
    alcs.alcs_spconv1x1_set_cfg(p, n, h, h, 0, dict(math_mode=4))
    x = torch.from_numpy(X).cuda()
    y = [torch.zeros((n, cout, h * h), device="cuda") for _ in range(2)]
    bias = y[0].view(-1)[:cout]                    # the first channel of the first layer's output
    st = alcs.alcs_stack_create([dict(w=p, x=x, y=y[0], n=n, h=h, wd=h, bias=torch.from_numpy(b).cuda(), flags=0),
                                 dict(w=p, x=x, y=y[1], n=n, h=h, wd=h, bias=bias, flags=0)], 0)
    for _ in range(3):
        y[0].zero_()
        alcs.alcs_stack_run(st, torch.cuda.current_stream())
    torch.cuda.synchronize()
    Y0, A0 = oracle.conv1x1(W, M, X, b, False, 4, want_scale=True)
    assert_parity(y[0].cpu().numpy(), Y0, A0, "f32")
    Y1, A1 = oracle.conv1x1(W, M, X, bias.cpu().numpy(), False, 4, want_scale=True)
    assert_parity(y[1].cpu().numpy(), Y1, A1, "f32")
    alcs.alcs_stack_destroy(st)


def test_rows_that_are_no_output_do_not_count_as_infinite(alcs):
    """One 7x7 image in a tile that has room for two: what the second one's rows hold is left over from the launch
    before, here infinities; a call must take as long as it does behind finite inputs (9 us, and 200 when every
    item was searched for the input that is not there)."""
    import torch
    n, cin, h, g = 2, 1024, 7, 8
    W, M, X, _ = _case(6, n, cin, 64, h * h, g, 0.5, np.float16)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    st, cfg = torch.cuda.current_stream(), dict(math_mode=4)
    bad = torch.full((n, cin, h * h), float("inf"), dtype=torch.float16, device="cuda")
    x, y2, y = torch.from_numpy(X).cuda(), torch.empty((n, 64, h * h), dtype=torch.float16, device="cuda"), torch.empty((1, 64, h * h), dtype=torch.float16, device="cuda")

    def us(first):
        best = 1e9
        for _ in range(5):
            alcs.alcs_spconv1x1(p, first, y2, n, h, h, None, 0, st, cfg)
            torch.cuda.synchronize()
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(10):
                alcs.alcs_spconv1x1(p, x, y, 1, h, h, None, 0, st, cfg)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]) * 100)
        return best

    us(x)
    assert us(bad) < 3 * us(x) + 20
    Yref, A = oracle.conv1x1(W, M, X[:1], None, False, g, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f16")


def _modes(alcs, sparsity, n, cin, cout, h, g, dtype=np.float32):
    W, M, _, _ = _case(1, 1, cin, cout, 1, g, 1.0 - sparsity, dtype)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    return alcs.alcs_spconv1x1_plan(p, n, h, h, 0)["math_mode"]


def test_sparse_layers_leave_the_dense_tiles_to_the_dense_ones(alcs):
    """The tcgen05 kernel's time hardly depends on the density, the CUDA cores' does: 92 us against 49 for 2048 -> 2048
    at 7x7, batch 32, 5 % kept, and 92 against 220 with half of the blocks kept."""
    assert _modes(alcs, 0.95, 32, 2048, 2048, 7, 4) == 1
    assert _modes(alcs, 0.5, 32, 2048, 2048, 7, 4) == 4
    assert _modes(alcs, 0.8, 64, 512, 512, 14, 4) == 4
    assert _modes(alcs, 0.5, 64, 512, 512, 14, 8, np.float16) == 4


# n, cin, cout, h, wd, g, stride, residual, density: strided rows of 8-byte copies and residuals that the staged kernels take
# sooner than plain layers, of every element type's path
@pytest.mark.parametrize("n,cin,cout,h,wd,g,stride,residual,density", [(8, 512, 512, 14, 14, 4, 2, False, 0.2), (32, 256, 512, 14, 14, 4, 3, True, 0.03),
                                                                      (64, 32, 64, 56, 56, 8, 1, True, 0.2), (4, 1024, 256, 14, 14, 1, 2, True, 0.03)])
@pytest.mark.parametrize("dtype", [np.float32, np.float16])
def test_planned_strided_and_residual_layers(alcs, n, cin, cout, h, wd, g, stride, residual, density, dtype):
    import torch
    W, M, X, b = _case(n + stride, n, cin, cout, h * wd, g, density, dtype)
    oh, ow = -(-h // stride), -(-wd // stride)
    R = rng.normal(6, 5, n * cout * oh * ow).reshape(n, cout, oh * ow).astype(dtype) if residual else None
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    xd, bd, rd = torch.from_numpy(X).cuda(), torch.from_numpy(b).cuda(), None if R is None else torch.from_numpy(R).cuda()
    Yref, A = oracle.conv1x1_ex(W, M, X.reshape(n, cin, h, wd), b, R, True, g, stride, want_scale=True)
    y = torch.full((n, cout, oh * ow), float("nan"), dtype=xd.dtype, device="cuda")
    alcs.alcs_spconv1x1_ex(p, xd, y, n, h, wd, stride, bd, rd, alcs.ALCS_RELU, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), Yref, A, "f32" if dtype == np.float32 else "f16")
    stack = alcs.alcs_stack_create([dict(w=p, x=xd, y=y, n=n, h=h, wd=wd, bias=bd, flags=alcs.ALCS_RELU, residual=rd, stride=stride)], 0)
    y.fill_(float("nan"))
    alcs.alcs_stack_run(stack, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), Yref, A, "f32" if dtype == np.float32 else "f16")
    alcs.alcs_stack_destroy(stack)


def _conv2d(alcs, p, X, b, cout, k, stride, pad, cfg=None):
    import torch
    n, cin, h, w = X.shape
    oh, ow = (h + 2 * pad - k[0]) // stride + 1, (w + 2 * pad - k[1]) // stride + 1
    y = torch.full((n, cout, oh, ow), float("nan"), device="cuda")
    alcs.alcs_spconv2d(p, torch.from_numpy(X).cuda(), y, n, cin, h, w, k[0], k[1], stride, pad, torch.from_numpy(b).cuda(), 0,
                       torch.cuda.current_stream(), cfg)
    torch.cuda.synchronize()
    return y.cpu().numpy()


_CONV_CFG = ("positions_per_lane", "strip_rows", "row_groups", "chunk_channels", "images_per_item")


# n, cin, cout, h, w, kh, kw, stride, pad: patches of one and of several images, rows copied by 16, 8 and 4 bytes, channel
# blocks with a remainder, borders on every side; dense enough for the tensor cores to be chosen
@pytest.mark.parametrize("n,cin,cout,h,w,kh,kw,stride,pad", [(8, 40, 160, 14, 14, 3, 3, 1, 1), (100, 65, 150, 9, 8, 3, 3, 2, 1), (4, 129, 300, 7, 7, 3, 3, 1, 1),
                                                            (12, 24, 130, 28, 30, 1, 3, 1, 1), (3, 100, 136, 12, 12, 5, 5, 1, 2), (8, 130, 160, 11, 8, 1, 1, 1, 0)])
def test_dense_kxk_layers_on_the_tensor_cores_and_sparse_ones_not(alcs, n, cin, cout, h, w, kh, kw, stride, pad):
    g, X = 1, rng.normal(n + cin, 2, n * cin * h * w).reshape(n, cin, h, w).astype(np.float32)
    for density in (1.0, 0.005):
        W, M, _, b = _case(n + cin + h, n, cin * kh * kw, cout, 1, g, density)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
        plan = alcs.alcs_spconv2d_plan(p, n, cin, h, w, kh, kw, stride, pad)
        cores = _conv2d(alcs, p, X, b, cout, (kh, kw), stride, pad, {k: plan[k] for k in _CONV_CFG})
        Y = _conv2d(alcs, p, X, b, cout, (kh, kw), stride, pad)
        Yref, A = oracle.conv2d(W.reshape(cout, cin, kh, kw), M, X, b, False, g, stride, pad, want_scale=True)
        assert_parity(cores, Yref, A, "f32")
        assert_parity(Y, Yref, A, "f32")
        # (the kernels differ in the order of their sums, so the bits show which one ran)
        if density == 1.0:
            assert not np.array_equal(Y, cores)


@pytest.mark.parametrize("n,cin,cout,h", [(1, 512, 512, 7), (16, 96, 96, 14)])
def test_kxk_layer_under_capture(alcs, n, cin, cout, h):
    """The first takes split columns, whose partial sums are the graph's own memory; replays see new inputs."""
    import torch
    g = 4
    W, M, _, b = _case(n + cin, n, cin * 9, cout, 1, g, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    X = rng.normal(3, 2, 2 * n * cin * h * h).reshape(2, n, cin, h, h).astype(np.float32)
    x, y, bd, side = torch.from_numpy(X[0]).cuda(), torch.zeros((n, cout, h, h), device="cuda"), torch.from_numpy(b).cuda(), torch.cuda.Stream()
    call = lambda: alcs.alcs_spconv2d(p, x, y, n, cin, h, h, 3, 3, 1, 1, bd, 0, side)
    side.wait_stream(torch.cuda.current_stream())
    call()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        call()
    for i in (1, 0, 1):
        x.copy_(torch.from_numpy(X[i]))
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        Yref, A = oracle.conv2d(W.reshape(cout, cin, 3, 3), M, X[i], b, False, g, 1, 1, want_scale=True)
        assert_parity(y.cpu().numpy(), Yref, A, "f32")


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("residual", [False, True])
def test_mostly_empty_channel_tiles(alcs, dtype, residual):
    """Tiles that keep nothing are bias and residual alone, for channel counts that do not end on four, and beside tiles
    that keep something, in and out of order of length."""
    import torch
    n, cin, cout, h, g = 3, 60, 158, 14, 2
    W, M, X, b = _case(5, n, cin, cout, h * h, g, 0.5, dtype)
    M[8:] = 0
    M[70, 3] = 1
    R = rng.normal(6, 5, n * cout * h * h).reshape(n, cout, h * h).astype(dtype)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    for tiles in (2, 5, 10):
        y = torch.full((n, cout, h * h), float("nan"), dtype=torch.from_numpy(X).dtype, device="cuda")
        alcs.alcs_spconv1x1_ex(p, torch.from_numpy(X).cuda(), y, n, h, h, 1, torch.from_numpy(b).cuda(), torch.from_numpy(R).cuda() if residual else None,
                               alcs.ALCS_RELU, torch.cuda.current_stream(), dict(math_mode=4, row_groups=tiles))
        torch.cuda.synchronize()
        Yref, A = oracle.conv1x1_ex(W, M, X.reshape(n, cin, h, h), b, R if residual else None, True, g, 1, want_scale=True)
        assert_parity(y.cpu().numpy(), Yref, A, "f32" if dtype == np.float32 else "f16")


def test_tuner_lists_what_an_untuned_call_may_run(alcs):
    """The planner considers the small-problem kernel for up to 64 images; so must the list that the tuner times (which is
    also where a configuration that names the kernel alone looks for its shape)."""
    import torch
    n, cin, cout, h, g = 24, 57, 48, 14, 16
    W, M, X, b = _case(3, n, cin, cout, h * h, g, 0.1)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    x, y, st = torch.from_numpy(X).cuda(), torch.empty((n, cout, h * h), device="cuda"), torch.cuda.current_stream()
    alcs.alcs_spconv1x1(p, x, y, n, h, h, None, 0, st, dict(math_mode=3))
    torch.cuda.synchronize()
    Yref, A = oracle.conv1x1(W, M, X, None, False, g, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f32")
    alcs.alcs_spconv1x1_tune(p, x, y, n, h, h, None, 0, st)
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), Yref, A, "f32")


def test_stack_of_tuned_layers_is_still_one_launch(alcs):
    """A layer tuned by itself may run otherwise in a stack: 13 layers of one image, tuned one by one, took 63 us in launches
    of their own against 23 in one.  A configuration that was set holds."""
    import torch
    layers, keep, st = [], [], torch.cuda.current_stream()
    for i, (cin, cout, h) in enumerate([(128, 256, 28), (256, 256, 28), (512, 512, 14), (512, 512, 14), (512, 1024, 7), (1024, 1024, 7)]):
        W, M, X, b = _case(90 + i, 1, cin, cout, h * h, 4, 0.2)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
        x, y, bd = torch.from_numpy(X).cuda(), torch.empty((1, cout, h * h), device="cuda"), torch.from_numpy(b).cuda()
        alcs.alcs_spconv1x1_tune(p, x, y, 1, h, h, bd, alcs.ALCS_RELU, st)
        layers.append(dict(w=p, x=x, y=y, n=1, h=h, wd=h, bias=bd, flags=alcs.ALCS_RELU))
        keep.append(oracle.conv1x1(W, M, X, b, True, 4, want_scale=True))
    stack = alcs.alcs_stack_create(layers, 0)
    assert {alcs.alcs_stack_layer_cfg(stack, i)["math_mode"] for i in range(len(layers))} == {4}
    alcs.alcs_stack_run(stack, st)
    torch.cuda.synchronize()
    for L, (Yref, A) in zip(layers, keep):
        assert_parity(L["y"].cpu().numpy(), Yref, A, "f32")
    alcs.alcs_stack_destroy(stack)
    alcs.alcs_spconv1x1_set_cfg(layers[2]["w"], 1, 14, 14, alcs.ALCS_RELU, dict(math_mode=3, pixels_per_lane=2, warps=4))
    stack = alcs.alcs_stack_create(layers, 0)
    assert alcs.alcs_stack_layer_cfg(stack, 2)["math_mode"] == 3
    alcs.alcs_stack_destroy(stack)


def test_tuning_releases_the_expanded_weights_that_lost(alcs):
    """25 MB for every width of a 2048 x 2048 layer in fp32, eight widths tried; forms that were there before stay."""
    import torch
    st, g = torch.cuda.current_stream(), 4

    def layer(n, cin, cout, h):
        W, M, X, _ = _case(3, n, cin, cout, h * h, g, 0.5)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
        return p, W, M, X, torch.from_numpy(X).cuda(), torch.empty((n, cout, h * h), device="cuda")

    p, *_, x, y = layer(4, 256, 256, 14)
    alcs.alcs_spconv1x1_tune(p, x, y, 4, 14, 14, None, 0, st)          # (loads the kernels that are timed)
    p, W, M, X, x, y = layer(4, 2048, 2048, 14)
    alcs.alcs_spconv1x1(p, x, y, 4, 14, 14, None, 0, st, dict(math_mode=4, row_groups=16))
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        alcs.alcs_spconv1x1(p, x, y, 4, 14, 14, None, 0, side, dict(math_mode=4, row_groups=16))
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    alcs.alcs_spconv1x1_tune(p, x, y, 4, 14, 14, None, 0, st)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < 80 << 20
    Yref, A = oracle.conv1x1(W, M, X, None, False, g, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f32")
    y.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert_parity(y.cpu().numpy(), Yref, A, "f32")


def test_very_large_matrices_are_not_expanded(alcs):
    """67 million weights, a thousandth of them kept, would take 400 MB as dense tiles: by default they stay as they are."""
    import torch
    n, c, h, g = 4, 8208, 7, 4
    M = (rng.uniform01(1, 3, c // g * c) < 0.001).astype(np.uint8).reshape(c // g, c)
    W = np.repeat(rng.normal(1, 1, c).astype(np.float32)[None, :], c, axis=0)
    X = rng.normal(1, 2, n * c * h * h).reshape(n, c, h * h).astype(np.float32)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    y, x = torch.empty((n, c, h * h), device="cuda"), torch.from_numpy(X).cuda()
    before = torch.cuda.mem_get_info()[0]
    alcs.alcs_spconv1x1(p, x, y, n, h, h, None, 0, torch.cuda.current_stream())
    assert alcs.alcs_spconv1x1_plan(p, n, h, h, 0)["math_mode"] != 4
    y2 = torch.empty((n, c, h, h), device="cuda")
    alcs.alcs_spconv2d(p, x, y2, n, c, h, h, 1, 1, 1, 0, None, 0, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < 350 << 20
    idx = np.arange(0, y.numel(), 997, dtype=np.int64)
    Yref = oracle.conv1x1_points(W, M, X, idx)
    Yref, A = Yref if isinstance(Yref, tuple) else (Yref, None)
    for t in (y, y2):
        d = np.abs(t.cpu().numpy().reshape(-1)[idx].astype(np.float64) - Yref)
        assert (d <= TOL["f32"] * (A if A is not None else np.abs(Yref).max())).all()


def test_forms_of_the_expanded_weights_are_bounded(alcs):
    """Calls of many batch sizes share a few forms: 14 MB each for 512 x 512 x 3 x 3."""
    import torch
    cin, cout, h, g = 512, 512, 7, 4
    W, M, _, _ = _case(3, 1, cin * 9, cout, 1, g, 0.5)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    X = rng.normal(4, 2, 64 * cin * h * h).reshape(64, cin, h, h).astype(np.float32)
    x, y, st = torch.from_numpy(X).cuda(), torch.empty((64, cout, h, h), device="cuda"), torch.cuda.current_stream()
    call = lambda n: alcs.alcs_spconv2d(p, x, y, n, cin, h, h, 3, 3, 1, 1, None, 0, st)
    call(1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for n in list(range(2, 64)) + [64]:
        call(n)
    torch.cuda.synchronize()
    # three more forms, and what the pool of the partial sums keeps (64 MB)
    assert before - torch.cuda.mem_get_info()[0] < (3 * 15 + 64 + 16) << 20
    Yref, A = oracle.conv2d(W.reshape(cout, cin, 3, 3), M, X[-2:], None, False, g, 1, 1, want_scale=True)
    assert_parity(y[-2:].cpu().numpy(), Yref, A, "f32")
