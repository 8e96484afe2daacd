"""Which kernel a call is given, and what it does there: calls at the edge of what the tcgen05 kernel takes must run on
another kernel (or be refused), and give what the oracle gives."""
import numpy as np
import pytest

import oracle
from alcs_workloads import rng
from gpu_util import TOL, assert_parity, check_layer

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
