"""Grouped launches at the edges of their tiles against the CPU oracle: maps whose pixels end inside a tile, filter tiles that end
inside a block of 64, several output buffers and a single one, tiles shared by two members, maps shared between slots."""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

TOL_BF16 = 2e-2  # max|err| / max|ref| per row, as in the other bf16 parity tests


# family, resolution (72 -> 18x18, 9x9, 5x5, 3x3 maps; 136 -> 34, 17, 9, 5; 224 -> 56 .. 7), images per query, queries, wave, in flight
@pytest.mark.parametrize("family,res,batch,n,wave,conc", [
    ("resnet", 72, 1, 5, 4, 2), ("resnet", 136, 1, 7, 7, 1), ("resnet", 72, 3, 4, 3, 2), ("resnet", 224, 1, 3, 2, 2), ("resnet", 40, 2, 3, 3, 1),
    ("mbv3", 72, 1, 5, 4, 2), ("mbv3", 104, 2, 3, 3, 1),
])
def test_waves_at_tile_edges(family, res, batch, n, wave, conc):
    fam = {"resnet": wl.RESNET, "mbv3": wl.MBV3}[family]
    _, onet, gnet = gu.nets(fam, True)
    cfgs = wl.uniform_stream(fam, n - 2, seed=res) + [wl.extreme_cfg(fam, False), wl.extreme_cfg(fam, True)]
    xs = wl.make_inputs(n, batch, res, seed=7, bf16=True)
    d_in = gu.to_device(xs.reshape(n * batch, res, res, 3), True)
    out = torch.full((n * batch, 1000), float("nan"), dtype=torch.float32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    opts = sgs.StreamOpts(cache_enabled=1, window_q=2, record_latency=0, concurrency=conc, wave=wave)
    for _ in range(2):  # (the second time with whatever the first left in the padding of its buffers)
        gnet.stream_run(cfgs, d_in.data_ptr(), batch, res, out.data_ptr(), opts, stream.cuda_stream)
    got = out.cpu().numpy().reshape(n, batch, 1000)
    assert np.all(np.isfinite(got))
    for t in range(n):
        ref = onet.forward(cfgs[t], xs[t], oracle.BF16_STORE)
        assert gu.rel_err(got[t], ref) <= TOL_BF16, t
    assert sgs.device_status() == 0


def test_single_query_of_many_images_equals_the_checker():
    # 16 images of 224x224: the layers with two tiles for every SM run on the grouped kernel, the others on the latency kernel;
    # with the cached SubGraph's hints on (their table is read by the kernel) and off
    _, onet, gnet = gu.nets(wl.RESNET, True)
    batch, res, n = 16, 224, 3
    cfgs = wl.markov_stream(n, seed=3)
    xs = wl.make_inputs(n, batch, res, seed=8, bf16=True)
    d_in = gu.to_device(xs.reshape(n * batch, res, res, 3), True)
    out = torch.zeros((2, n * batch, 1000), dtype=torch.float32, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for i, cache in enumerate((0, 1)):
        opts = sgs.StreamOpts(cache_enabled=cache, window_q=1, use_graphs=1, record_latency=0, concurrency=1, wave=0)
        for _ in range(2):
            gnet.stream_run(cfgs, d_in.data_ptr(), batch, res, out[i].data_ptr(), opts, stream.cuda_stream)
    got = out.cpu().numpy()
    np.testing.assert_array_equal(got[0], got[1])
    for t, b in ((0, 0), (1, 7), (2, 15)):
        ref = onet.forward(cfgs[t], xs[t][b:b + 1], oracle.BF16_STORE)
        assert gu.rel_err(got[0][t * batch + b:t * batch + b + 1], ref) <= TOL_BF16
    assert sgs.device_status() == 0
