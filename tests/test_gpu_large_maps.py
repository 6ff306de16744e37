"""MobileNetV3-shaped SubNets at resolutions where the maps of some squeeze-and-excite blocks are too large for the one-launch
kernel: those blocks run as pool, gate and scale, in single queries, waves (also where members of one wave differ in it) and the
persistent kernel."""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# bf16 maps above about 50x50 with 240 channels (resolution 400), fp32 above 35x35
@pytest.mark.parametrize("res,bf16", [(512, True), (416, True), (320, False)])
def test_single_queries(res, bf16):
    _, onet, gnet = gu.nets(wl.MBV3, bf16)
    cfg = wl.extreme_cfg(wl.MBV3, True)
    x = wl.make_inputs(1, 1, res, seed=res, bf16=bf16)[0]
    ref = onet.forward(cfg, x, mode=oracle.BF16_STORE if bf16 else oracle.FP32)
    assert gu.rel_err(gu.gpu_forward(gnet, cfg, x, bf16), ref) <= (2e-2 if bf16 else 1e-4)


@pytest.mark.parametrize("res", [416, 512])
def test_streams(res):
    # at 416 the blocks of 160 and less channels of a stage fit the kernel, those of 240 do not
    _, _, gnet = gu.nets(wl.MBV3, True)
    n = 7
    cfgs = wl.uniform_stream(wl.MBV3, n - 2, seed=5) + [wl.extreme_cfg(wl.MBV3, False), wl.extreme_cfg(wl.MBV3, True)]
    x = gu.to_device(wl.make_inputs(n, 1, res, seed=1, bf16=True).reshape(n, res, res, 3), True)
    st = torch.cuda.Stream()
    runs = {}
    for wave, persistent in ((0, 0), (4, 0), (0, 1)):
        y = torch.zeros(n, 1000, device="cuda")
        torch.cuda.synchronize()
        gnet.stream_run(cfgs, x.data_ptr(), 1, res, y.data_ptr(),
                        sgs.StreamOpts(cache_enabled=1, window_q=4, wave=wave, concurrency=2 if wave else 1, persistent=persistent), st.cuda_stream)
        runs[wave, persistent] = y.cpu().numpy()
    assert np.isfinite(runs[0, 0]).all() and gu.rel_err(runs[4, 0], runs[0, 0]) <= 2e-2 and gu.rel_err(runs[0, 1], runs[0, 0]) <= 2e-2


def test_plans_made_under_another_convolution_option():
    # the order of a wave's layers is worked out once: also when the first plans of a handle were made without tensor cores
    net = sgs.SuperNet(wl.RESNET, wl.make_blob(wl.RESNET, seed=0, bf16_weights=True), sgs.SGS_BF16)
    cfg, x = wl.extreme_cfg(wl.RESNET, False), wl.make_inputs(1, 1, 64, seed=1, bf16=True)[0]
    net.set_option("conv_impl", 1)
    plain = gu.gpu_forward(net, cfg, x, True)
    net.set_option("conv_impl", 0)
    tc = gu.gpu_forward(net, cfg, x, True)
    net.close()
    assert gu.rel_err(tc, plain) <= 2e-2
