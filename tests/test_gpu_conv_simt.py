"""GPU parity of the CUDA-core convolution (sgs_conv2d_sliced, impl 1) at the edges of its tiles, its reduction steps of 32,
its cluster splits and both copy widths, against a plain fp32 convolution."""
import pytest
import torch

import paper_2306_17266_b200 as sgs

pytestmark = pytest.mark.gpu

# N, H, W, Cmax, C, Kmax, K, R, k, stride, act, residual
CASES = [
    (1, 1, 1, 8, 4, 8, 4, 1, 1, 1, 0, False),          # one pixel, one step of four channels
    (1, 5, 5, 3, 3, 16, 10, 7, 7, 1, 1, False),        # single-element copies (3 channels), K not a multiple of 4
    (2, 9, 7, 12, 12, 24, 20, 3, 3, 2, 1, True),       # odd sizes at stride 2, 108-long reduction
    (1, 8, 8, 72, 64, 72, 65, 3, 3, 1, 2, True),       # K one beyond a tile
    (1, 7, 9, 40, 33, 40, 31, 3, 1, 1, 0, True),       # centre tap of a stored 3x3, odd channel count
    (1, 4, 4, 368, 360, 64, 48, 3, 3, 1, 1, False),    # long reduction on few pixels: cluster of 8
    (3, 40, 40, 64, 56, 96, 88, 1, 1, 1, 1, True),     # many tiles, no split
    (1, 64, 65, 16, 16, 32, 24, 7, 5, 1, 0, False),    # centre 5x5 of a stored 7x7
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_cuda_core_convolution(case, dtype):
    N, H, W, Cmax, C, Kmax, K, R, k, stride, act, use_res = case
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(3)
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g)
    p, o = (k - 1) // 2, (R - k) // 2
    Ho, Wo = (H + 2 * p - k) // stride + 1, (W + 2 * p - k) // stride + 1
    x, w = rnd(N, H, W, C).to(td), (rnd(Kmax, R, R, Cmax) * 0.1).to(td)
    sc, sh = rnd(Kmax), rnd(Kmax)
    res = rnd(N, Ho, Wo, K).to(td) if use_res else None
    y = torch.full((N, Ho, Wo, K), 77.0, device="cuda", dtype=td)
    d = sgs.ConvDesc(N=N, H=H, W=W, C=C, K=K, Kmax=Kmax, Cmax=Cmax, R=R, k=k, stride=stride, act=act,
                     dtype=sgs.SGS_F32 if dtype == "f32" else sgs.SGS_BF16, impl=1)
    runs = []
    for _ in range(2):
        sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), sc.data_ptr(), sh.data_ptr(), res.data_ptr() if use_res else 0, y.data_ptr(),
                          torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        runs.append(y.clone())
    ws = w[:K, o:o + k, o:o + k, :C].permute(0, 3, 1, 2).double().cpu()
    ref = torch.nn.functional.conv2d(x.permute(0, 3, 1, 2).double().cpu(), ws, stride=stride, padding=p).permute(0, 2, 3, 1)
    ref = ref * sc[:K].double().cpu() + sh[:K].double().cpu() + (res.double().cpu() if use_res else 0)
    ref = torch.relu(ref) if act == 1 else torch.nn.functional.hardswish(ref) if act == 2 else ref
    err = (y.double().cpu() - ref).abs().max().item() / ref.abs().max().item()
    assert err <= (2e-6 if dtype == "f32" else 5e-3)
    assert torch.equal(runs[0], runs[1])
