"""GPU parity of the tcgen05 kernel (math_mode 4) against the oracle at the sizes where its tiles, chunks and
copies change: pixel tiles that end inside or between images, column chunks with remainders, channel tiles that
end in padding, every way X is brought in, and the merged launch of a stack's independent layers."""
import numpy as np
import pytest

import oracle
from alcs_workloads import rng
from gpu_util import assert_parity, check_layer

pytestmark = pytest.mark.gpu


def _case(seed, n, cin, cout, hw, g, density, dtype=np.float32):
    rows = (cout + g - 1) // g
    W = (rng.normal(seed, 1, cout * cin) * cin ** -0.5).reshape(cout, cin).astype(dtype)
    X = rng.normal(seed, 2, n * cin * hw).reshape(n, cin, hw).astype(dtype)
    M = (rng.uniform01(seed, 3, rows * cin) < density).astype(np.uint8).reshape(rows, cin)
    return W, M, X, (0.1 * rng.normal(seed, 4, cout)).astype(np.float32)


# n, cin, cout, h, wd, g, density: one channel and one pixel; 16-byte, 8-byte, 4-byte and single-element copies; whole
# images per tile with a rest; chunk remainders (cin 65, 129); channel tiles with padding (cout 130, 200); a column
# list (few kept columns); more items than SMs
SHAPES = [(1, 1, 1, 1, 1, 1, 1.0), (2, 40, 24, 10, 5, 4, 0.4), (3, 65, 130, 9, 9, 2, 0.5), (5, 64, 48, 7, 7, 8, 0.5),
          (3, 129, 200, 14, 14, 4, 0.3), (9, 256, 64, 4, 4, 8, 0.02), (2, 96, 16, 13, 6, 16, 0.5), (70, 80, 260, 16, 16, 4, 0.2)]


@pytest.mark.parametrize("dtype", [np.float32, np.float16])
@pytest.mark.parametrize("n,cin,cout,h,wd,g,density", SHAPES)
def test_shapes(alcs, n, cin, cout, h, wd, g, density, dtype):
    W, M, X, b = _case(n + cin + cout, n, cin, cout, h * wd, g, density, dtype)
    for tiles in {0, -(-cout // 16)}:
        check_layer(alcs, W, M, X, b, True, g, cfg=dict(math_mode=4, row_groups=tiles), h=h, wd=wd)
    check_layer(alcs, W, M, X, None, False, g, cfg=dict(math_mode=4), h=h, wd=wd, y_f32=dtype == np.float16)


@pytest.mark.parametrize("scale", [1e-30, 1.0, 1e30])
def test_fp32_operands_are_not_rounded(alcs, scale):
    """The three bfloat16 parts of an operand add up to it, over the exponent range, in X and in W."""
    n, cin, cout, hw, g = 2, 70, 32, 50, 4
    W, M, X, _ = _case(77, n, cin, cout, hw, g, 0.5)
    check_layer(alcs, W, M, (X * np.float32(scale)).astype(np.float32), None, False, g, cfg=dict(math_mode=4))
    check_layer(alcs, (W * np.float32(scale)).astype(np.float32), M, X, None, False, g, cfg=dict(math_mode=4))


def test_empty_and_skewed_rows(alcs):
    """Channel tiles that keep nothing (output = bias), and rows sorted by length into tiles with column lists."""
    n, cin, cout, hw, g = 3, 300, 256, 196, 4
    W, M, X, b = _case(5, n, cin, cout, hw, g, 0.05)
    M[3::2] = 0
    M[0] = 1
    for tiles in (2, 8, 16):
        check_layer(alcs, W, M, X, b, True, g, cfg=dict(math_mode=4, row_groups=tiles), h=14, wd=14)
    M[:] = 0
    check_layer(alcs, W, M, X, b, True, g, cfg=dict(math_mode=4), h=14, wd=14, exact=True)


@pytest.mark.parametrize("graph", [False, True])
def test_merged_stack(alcs, graph):
    """Independent layers run as one launch; a layer that reads another one's output must not be merged with it."""
    import torch
    dev = torch.device("cuda:0")
    shapes = [(2, 64, 96, 14, 14), (2, 96, 80, 14, 14), (2, 128, 48, 7, 7), (2, 32, 160, 28, 28)]
    layers, keep = [], []
    for i, (n, cin, cout, h, wd) in enumerate(shapes):
        W, M, X, b = _case(40 + i, n, cin, cout, h * wd, 4, 0.3)
        p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
        x = layers[0]["y"] if i == 1 else torch.from_numpy(X).to(dev)       # layer 1 continues layer 0
        layers.append(dict(w=p, x=x, y=torch.full((n, cout, h * wd), float("nan"), device=dev), n=n, h=h, wd=wd,
                           bias=torch.from_numpy(b).to(dev), flags=alcs.ALCS_RELU))
        keep.append((W, M, X, b))
        if i != 1:
            alcs.alcs_spconv1x1_set_cfg(p, n, h, wd, alcs.ALCS_RELU, dict(math_mode=4))
    alcs.alcs_spconv1x1_set_cfg(layers[1]["w"], 2, 14, 14, alcs.ALCS_RELU, dict(math_mode=4))
    st = alcs.alcs_stack_create(layers, alcs.ALCS_STACK_GRAPH if graph else 0)
    stream = torch.cuda.Stream()
    for _ in range(3):
        alcs.alcs_stack_run(st, stream)
    stream.synchronize()
    prev = None
    for i, (W, M, X, b) in enumerate(keep):
        Y = layers[i]["y"].cpu().numpy()
        Yref, A = oracle.conv1x1(W, M, prev if i == 1 else X, b, True, 4, want_scale=True)
        assert_parity(Y, Yref, A, "f32")
        prev = Y
    assert all(alcs.alcs_packed_status(L["w"]) == 0 for L in layers)
    alcs.alcs_stack_destroy(st)


# n, cin, cout, h, w, kh, kw, stride, pad: patches of one and of several images, rows copied by 16, 8 and 4 bytes,
# channel blocks with a remainder, fewer taps than steps per chunk, borders on every side, more slots than one item uses;
# the first two have few pixels and many channels, so that their columns are split
PATCHES = [(1, 200, 20, 7, 7, 3, 3, 1, 1), (2, 129, 150, 9, 8, 3, 3, 2, 1), (2, 16, 16, 5, 6, 3, 3, 1, 1), (5, 33, 40, 7, 7, 3, 3, 1, 1), (3, 20, 130, 14, 14, 3, 3, 2, 1), (2, 70, 24, 28, 30, 1, 3, 1, 1),
           (1, 17, 16, 9, 56, 5, 3, 2, 2), (9, 8, 12, 4, 3, 2, 2, 2, 0), (2, 130, 16, 11, 8, 1, 1, 1, 0)]


@pytest.mark.parametrize("n,cin,cout,h,w,kh,kw,stride,pad", PATCHES)
def test_patch_staging(alcs, n, cin, cout, h, w, kh, kw, stride, pad):
    import torch
    g, taps = 4, kh * kw
    W, M, _, b = _case(3 * n + cin + h, n, cin * taps, cout, 1, g, 0.4)
    X = rng.normal(n + cin, 2, n * cin * h * w).reshape(n, cin, h, w).astype(np.float32)
    oh, ow = (h + 2 * pad - kh) // stride + 1, (w + 2 * pad - kw) // stride + 1
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, g), 0)
    y = torch.full((n, cout, oh, ow), float("nan"), device="cuda:0")
    alcs.alcs_spconv2d(p, torch.from_numpy(X).cuda(), y, n, cin, h, w, kh, kw, stride, pad, torch.from_numpy(b).cuda(),
                       alcs.ALCS_RELU, torch.cuda.current_stream())
    torch.cuda.synchronize()
    Yref, A = oracle.conv2d(W.reshape(cout, cin, kh, kw), M, X, b, True, g, stride, pad, want_scale=True)
    assert_parity(y.cpu().numpy(), Yref, A, "f32")
    assert alcs.alcs_packed_status(p) == 0


@pytest.mark.parametrize("n,cin,cout,h", [(3, 64, 96, 28), (16, 128, 160, 14), (13, 61, 300, 7), (41, 96, 96, 7)])
def test_host_call_in_pieces(alcs, n, cin, cout, h):
    """Calls large enough to be cut into pieces, among them sizes whose pieces cannot start on 16-byte boundaries."""
    import torch
    W, M, X, b = _case(n + cin, n, cin, cout, h * h, 4, 0.3)
    p = alcs.alcs_packed_upload(alcs.alcs_pack(W, M, 4), 0)
    size = alcs.alcs_spconv1x1_host_workspace(p, n, h, h, alcs.ALCS_RELU)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda:0")
    xh, bh = torch.from_numpy(X).pin_memory(), torch.from_numpy(b).pin_memory()
    yh = torch.full((n, cout, h * h), float("nan")).pin_memory()
    stream = torch.cuda.Stream()
    for _ in range(3):
        alcs.alcs_spconv1x1_host(p, xh, yh, n, h, h, bh, alcs.ALCS_RELU, ws, size, stream)
    stream.synchronize()
    Yref, A = oracle.conv1x1(W, M, X, b, True, 4, want_scale=True)
    assert_parity(yh.numpy(), Yref, A, "f32")
