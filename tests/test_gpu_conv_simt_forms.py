"""CUDA-core convolution, both forms of its small tiles (few blocks, many short ones, many long ones) and folded batch norm that is not
16-byte aligned, against a plain convolution in 64 bits."""
import pytest
import torch

import paper_2306_17266_b200 as sgs

pytestmark = pytest.mark.gpu


# N, H, W, C, K, k, offset of scale and shift in elements
@pytest.mark.parametrize("N,H,W,C,K,k,off", [
    (1, 10, 10, 64, 72, 3, 0), (1, 10, 10, 64, 72, 3, 1), (1, 10, 10, 64, 70, 1, 3),   # one round
    (8, 48, 48, 16, 16, 3, 0), (8, 48, 48, 16, 32, 3, 2),                              # many blocks, five steps
    (6, 40, 40, 48, 48, 3, 0), (6, 40, 40, 48, 44, 3, 1),                              # many blocks, fourteen steps
])
def test_forms_of_the_small_tiles(N, H, W, C, K, k, off):
    g = torch.Generator(device="cuda").manual_seed(K + off)
    x = torch.randn(N, H, W, C, device="cuda", generator=g)
    w = torch.randn(K, k, k, C, device="cuda", generator=g) / (C * k * k) ** 0.5
    sc, sh = (torch.randn(K + off, device="cuda", generator=g)[off:] for _ in range(2))
    y = torch.full((N, H, W, K), 77.0, device="cuda")
    d = sgs.ConvDesc(N=N, H=H, W=W, C=C, K=K, Kmax=K, Cmax=C, R=k, k=k, stride=1, act=1, dtype=sgs.SGS_F32, impl=1)
    sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), sc.data_ptr(), sh.data_ptr(), 0, y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref = torch.nn.functional.conv2d(x.permute(0, 3, 1, 2).double().cpu(), w.permute(0, 3, 1, 2).double().cpu(), padding=(k - 1) // 2).permute(0, 2, 3, 1)
    ref = torch.relu(ref * sc.double().cpu() + sh.double().cpu())
    # (432 fp32 additions at most: some 20 roundings' worth of a result of the order of 1)
    assert (y.double().cpu() - ref).abs().max().item() / ref.abs().max().item() <= 2e-6
