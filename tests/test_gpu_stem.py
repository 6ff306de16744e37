"""Stem kernels (7x7 stride 2 with its max pool, 3x3 of both strides) through whole networks at the edges of their tiles: 17 x 7
convolution outputs around 8 x 3 pooled ones, 16 x 8 without a pool.  (The stem's map itself: test_gpu_layer_maps.py.)"""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

TOL_BF16 = 2e-2  # max|err| / max|ref| per row, as in the other bf16 parity tests


# odd and even images, maps that end inside a tile, at its end and one beyond (resnet pools to 8 a tile across, 3 down: 33 -> 17 -> 9)
@pytest.mark.parametrize("family,res,batch", [
    ("resnet", 64, 1), ("resnet", 75, 2), ("resnet", 97, 1), ("resnet", 32, 3), ("resnet", 130, 1),
    ("mbv3", 34, 2), ("mbv3", 64, 1), ("mbv3", 70, 1), ("mbv3", 33, 2), ("mbv3", 71, 1), ("tiny", 32, 1), ("tiny", 24, 3), ("tiny", 41, 2),
])
def test_networks_behind_the_stem(family, res, batch):
    fam = {"resnet": wl.RESNET, "mbv3": wl.MBV3, "tiny": wl.TINY}[family]
    _, onet, gnet = gu.nets(fam, True)
    stream = torch.cuda.Stream()
    for cfg in [wl.extreme_cfg(fam, False), wl.extreme_cfg(fam, True)] + wl.uniform_stream(fam, 2, seed=res):
        xs = wl.make_inputs(1, batch, res, seed=9, bf16=True)
        d_in = gu.to_device(xs.reshape(batch, res, res, 3), True)
        # an image that starts at an odd 2-byte address
        shifted = torch.empty(d_in.numel() + 1, dtype=torch.bfloat16, device="cuda")
        shifted[1:] = d_in.reshape(-1)
        out = torch.full((2, batch, gnet.n_classes), float("nan"), dtype=torch.float32, device="cuda")
        arr = wl.cfg_array([cfg])
        torch.cuda.synchronize()
        gnet.subnet_run(arr[0], d_in.data_ptr(), batch, res, out[0].data_ptr(), stream.cuda_stream)
        if fam != wl.TINY:  # (a 12-filter stem is a direct convolution)
            gnet.subnet_run(arr[0], shifted.data_ptr() + 2, batch, res, out[1].data_ptr(), stream.cuda_stream)
        torch.cuda.synchronize()
        ref = onet.forward(cfg, xs[0], oracle.BF16_STORE)
        got = out.cpu().numpy()
        assert gu.rel_err(got[0], ref) <= TOL_BF16
        if fam != wl.TINY:
            np.testing.assert_array_equal(got[0], got[1])
    assert sgs.device_status() == 0
