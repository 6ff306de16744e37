"""GPU parity of the fused squeeze-excite block (through whole MobileNetV3-shaped SubNets: its pixel shares, its ragged last
share, maps smaller than its cluster), of the linear layer at the edges of its row and output groups, and of the
tensor-core convolution at stride 2 on odd sizes."""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from paper_2306_17266_b200.binding import SGS_AUX_LINEAR
from tests.gpu_util import gpu_forward, nets, rel_err

pytestmark = pytest.mark.gpu


# (resolution, images): stage maps from 1x1 (fewer pixels than blocks) to 30x30
@pytest.mark.parametrize("res,batch", [(16, 2), (40, 3), (72, 1), (240, 1)])
@pytest.mark.parametrize("bf16", [True, False])
def test_squeeze_excite_block(res, batch, bf16):
    blob, onet, gnet = nets(wl.MBV3, bf16)
    x = wl.make_inputs(1, batch, res, seed=res, bf16=bf16)[0]
    cfg = wl.uniform_stream(wl.MBV3, 1, seed=res + batch)[0]
    ref = onet.forward(cfg, x, mode=oracle.BF16_STORE if bf16 else oracle.FP32)
    assert rel_err(gpu_forward(gnet, cfg, x, bf16), ref) <= (2e-2 if bf16 else 1e-4)


@pytest.mark.parametrize("rows", [1, 2, 3, 8, 9, 17])
@pytest.mark.parametrize("K,C,ld", [(1, 8, 8), (5, 264, 272), (1003, 520, 520), (1000, 2048, 2048)])
def test_linear_rows(rows, K, C, ld):
    rng = np.random.default_rng(rows)
    w = wl.round_to_bf16(rng.standard_normal((K, ld)).astype(np.float32) * 0.05)
    b = rng.standard_normal(K).astype(np.float32)
    x = rng.standard_normal((rows, C)).astype(np.float32)
    dw, db, dx = torch.from_numpy(w).cuda().to(torch.bfloat16), torch.from_numpy(b).cuda(), torch.from_numpy(x).cuda()
    ref = x.astype(np.float64) @ w[:, :C].astype(np.float64).T + b
    for grouped in (False, True):  # one query of `rows` images; `rows` members of one image
        n, per = (rows, 1) if grouped else (1, rows)
        dy = [torch.full((per, K), 77.0, device="cuda") for _ in range(n)]
        dxs = [dx[i * per:(i + 1) * per].clone() for i in range(n)]
        d = [sgs.AuxDesc(kind=SGS_AUX_LINEAR, dtype=sgs.SGS_BF16, N=per, H=1, W=1, C=C, K=K, ld=ld, act=0)] * n
        a = [sgs.AuxArgs(x=dxs[i].data_ptr(), y=dy[i].data_ptr(), w=dw.data_ptr(), bias=db.data_ptr()) for i in range(n)]
        sgs.aux_op(d, a, grouped, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert np.abs(torch.cat(dy).cpu().numpy() - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("k", [1, 3, 5])
@pytest.mark.parametrize("N,H,W", [(1, 11, 11), (2, 2, 3), (3, 13, 8), (1, 55, 57)])
def test_stride_two_on_odd_sizes(N, H, W, k):
    g = torch.Generator(device="cuda").manual_seed(5)
    C, K, R = 72, 40, 5 if k == 5 else k
    x = torch.randn(N, H, W, C, device="cuda", generator=g).to(torch.bfloat16)
    w = (torch.randn(K + 8, R, R, C + 8, device="cuda", generator=g) * 0.05).to(torch.bfloat16)
    sc, sh = torch.rand(K + 8, device="cuda", generator=g) + 0.5, torch.randn(K + 8, device="cuda", generator=g)
    p = (k - 1) // 2
    ref = torch.nn.functional.conv2d(x.permute(0, 3, 1, 2).double().cpu(), w[:K, :, :, :C].permute(0, 3, 1, 2).double().cpu(), stride=2, padding=p)
    ref = torch.relu(ref.permute(0, 2, 3, 1) * sc[:K].double().cpu() + sh[:K].double().cpu())
    y = torch.full(ref.shape, 77.0, device="cuda", dtype=torch.bfloat16)
    d = sgs.ConvDesc(N=N, H=H, W=W, C=C, K=K, Kmax=K + 8, Cmax=C + 8, R=R, k=k, stride=2, act=1, dtype=sgs.SGS_BF16, impl=2)
    sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), sc.data_ptr(), sh.data_ptr(), 0, y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert (y.double().cpu() - ref).abs().max() <= 1e-2 * ref.abs().max()
