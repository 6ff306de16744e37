"""Depthwise, split-reduction and 8-bit kernels at the edges of their tiles, against fp32 PyTorch and the exact integer layer."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import oracle
import paper_2306_17266_b200 as sgs

pytestmark = pytest.mark.gpu


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _close(y, ref):
    assert sgs.device_status() == 0
    err = (y.float() - ref).abs().max().item() / ref.abs().max().item()
    assert err < 1e-2, err


# N, H, W, K, k, stride, act: narrow and wide strips (maps of 23, 24, 25 columns), one channel vector, ragged channel
# blocks, odd last row of a step, windows larger than the map, many row segments and whole columns
@pytest.mark.parametrize("N,H,W,K,k,stride,act", [
    (1, 1, 1, 8, 3, 1, 0), (1, 2, 3, 56, 7, 1, 1), (2, 7, 23, 72, 5, 1, 2), (1, 24, 24, 64, 3, 1, 1), (1, 25, 25, 136, 5, 1, 2),
    (3, 33, 49, 64, 7, 1, 0), (1, 47, 47, 40, 3, 2, 2), (2, 50, 50, 72, 5, 2, 1), (1, 13, 15, 200, 7, 2, 2), (64, 30, 57, 128, 5, 1, 2),
])
def test_depthwise_edges(N, H, W, K, k, stride, act):
    g = torch.Generator(device="cuda").manual_seed(K + k)
    x = torch.randn(N, H, W, K, device="cuda", generator=g).bfloat16()
    w = (torch.randn(7, 7, K + 8, device="cuda", generator=g) / k).bfloat16()
    scale, shift = torch.rand(K, device="cuda", generator=g) + 0.5, torch.randn(K, device="cuda", generator=g)
    o, p = (7 - k) // 2, (k - 1) // 2
    wk = w[o:o + k, o:o + k, :K].float().permute(2, 0, 1).unsqueeze(1)
    with torch.backends.cudnn.flags(enabled=False):
        ref = F.conv2d(x.float().permute(0, 3, 1, 2), wk.contiguous(), stride=stride, padding=p, groups=K).permute(0, 2, 3, 1)
    ref = ref * scale + shift
    ref = ref if act == 0 else ref.relu() if act == 1 else F.hardswish(ref)
    y = torch.empty(ref.shape, device="cuda", dtype=torch.bfloat16)
    desc = sgs.ConvDesc(N=N, H=H, W=W, C=1, K=K, Kmax=K + 8, Cmax=1, R=7, k=k, stride=stride, act=act, dtype=sgs.SGS_BF16, depthwise=1)
    sgs.conv2d_sliced(desc, x.data_ptr(), w.data_ptr(), scale.data_ptr(), shift.data_ptr(), 0, y.data_ptr(), _stream())
    torch.cuda.synchronize()
    _close(y, ref.contiguous())


# N, H, W, C, K, k, stride, residual: reductions over clusters of 2, 4 and 8 blocks, tiles with fewer rows than a block's
# share, filters beyond the last full tile at a half and a quarter of a tile
@pytest.mark.parametrize("N,H,W,C,K,k,stride,residual", [
    (1, 7, 7, 640, 512, 1, 1, True), (1, 7, 7, 512, 24, 3, 1, False), (1, 14, 14, 264, 248, 3, 2, True), (1, 3, 5, 1304, 72, 1, 1, False),
    (1, 28, 28, 136, 96, 3, 1, True), (16, 28, 28, 64, 152, 1, 1, True), (16, 28, 28, 72, 176, 3, 1, False), (1, 1, 1, 2048, 8, 1, 1, False),
])
def test_split_reduction_and_narrow_tiles(N, H, W, C, K, k, stride, residual):
    g = torch.Generator(device="cuda").manual_seed(C + K)
    x = torch.randn(N, H, W, C, device="cuda", generator=g).bfloat16()
    w = (torch.randn(K + 8, k, k, C + 8, device="cuda", generator=g) / (C * k * k) ** 0.5).bfloat16()
    scale, shift = torch.rand(K, device="cuda", generator=g) + 0.5, torch.randn(K, device="cuda", generator=g)
    # (unfolded product: fp32 without the reduced-precision convolution modes)
    cols = F.unfold(x.float().permute(0, 3, 1, 2), k, padding=(k - 1) // 2, stride=stride)
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1
    ref = (w[:K, :, :, :C].float().permute(0, 3, 1, 2).reshape(K, -1).double() @ cols.double()).float()
    ref = ref.reshape(N, K, Ho, Wo).permute(0, 2, 3, 1) * scale + shift
    res = torch.randn(ref.shape, device="cuda", generator=g).bfloat16() if residual else None
    ref = (ref + res.float() if residual else ref).relu()
    y = torch.empty(ref.shape, device="cuda", dtype=torch.bfloat16)
    desc = sgs.ConvDesc(N=N, H=H, W=W, C=C, K=K, Kmax=K + 8, Cmax=C + 8, R=k, k=k, stride=stride, act=1, dtype=sgs.SGS_BF16, depthwise=0)
    sgs.conv2d_sliced(desc, x.data_ptr(), w.data_ptr(), scale.data_ptr(), shift.data_ptr(), res.data_ptr() if residual else 0, y.data_ptr(),
                      _stream())
    torch.cuda.synchronize()
    _close(y, ref.contiguous())


# the ends of the 32-bit zero points: sums that only 64 bits hold
@pytest.mark.parametrize("zy", [-2 ** 31, -2 ** 28, 2 ** 28, 2 ** 31 - 1])
@pytest.mark.parametrize("relu", [False, True])
def test_int8_zero_point_ranges(zy, relu):
    _requantise(2, 4, False, False, 72, zy=zy, relu=relu)


# shifts on both sides of what 32-bit requantisation takes, biases that only 64-bit sums hold, the widest shift
@pytest.mark.parametrize("shift_lo,shift_hi,big_bias,residual,K", [(0, 2, False, True, 176), (2, 3, False, True, 176), (1, 4, True, False, 72),
                                                                   (2, 4, True, True, 136), (31, 32, False, False, 40)])
def test_int8_requantisation_ranges(shift_lo, shift_hi, big_bias, residual, K):
    _requantise(shift_lo, shift_hi, big_bias, residual, K)


def _requantise(shift_lo, shift_hi, big_bias, residual, K, zy=100, relu=False):
    rng = np.random.default_rng(shift_lo + K)
    N, H, C = 2, 9, 64
    w = rng.integers(-2, 3, (K, C, 1, 1)).astype(np.int8)
    x = rng.integers(0, 8, (N, H, H, C)).astype(np.uint8)
    mult = rng.integers(2 ** 30, 2 ** 31, K).astype(np.int32)
    shift = rng.integers(shift_lo, shift_hi, K).astype(np.int32)
    bias = rng.integers(-30, 30, K).astype(np.int32)
    if big_bias:
        bias[::3] = rng.choice([-2 ** 31, -2 ** 29, 2 ** 29, 2 ** 31 - 1], bias[::3].shape).astype(np.int32)
    res = rng.integers(0, 256, (N, H, H, K)).astype(np.uint8) if residual else None
    ref = oracle.layer_conv_i8(w, x, C, K, 1, 1, mult, shift, bias, zx=0, zy=zy, relu=relu, res=res, zr=128, res_mult=1932735283, res_shift=1,
                               y_signed=False)
    dx, dw, dm, ds, db = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w.transpose(0, 2, 3, 1), mult, shift, bias))
    dr = torch.from_numpy(res).cuda() if residual else None
    dy = torch.empty(ref.shape, dtype=torch.uint8, device="cuda")
    desc = sgs.ConvI8Desc(N=N, H=H, W=H, C=C, K=K, Kmax=K, Cmax=C, R=1, k=1, stride=1, relu=int(relu), zy=zy, zr=128, res_mult=1932735283, res_shift=1)
    sgs.conv2d_sliced_i8(desc, dx.data_ptr(), dw.data_ptr(), dm.data_ptr(), ds.data_ptr(), db.data_ptr(), dr.data_ptr() if residual else 0,
                         dy.data_ptr(), _stream())
    torch.cuda.synchronize()
    assert sgs.device_status() == 0
    np.testing.assert_array_equal(dy.cpu().numpy(), ref)
