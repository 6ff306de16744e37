"""Calls under stream capture: what only enqueues kernels can be captured once its set-up is done and gives the same on replay;
what has to synchronise the stream refuses it and leaves the handle as it was."""
import numpy as np
import pytest
import torch

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from paper_2306_17266_b200.binding import SGS_AUX_LINEAR, SGS_EINVAL
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _conv(kind):
    """(inputs kept alive, output, call on a stream) of one layer."""
    g = torch.Generator(device="cuda").manual_seed(3)
    dt = torch.float32 if kind == "f32" else torch.bfloat16
    depthwise = kind == "depthwise"
    N, H, C, K, k = (2, 40, 64, 64, 7) if depthwise else (1, 14, 256, 192, 3)
    x = torch.randn(N, H, H, C, device="cuda", generator=g).to(dt)
    w = (torch.randn(k, k, K, device="cuda", generator=g) if depthwise else torch.randn(K, k, k, C, device="cuda", generator=g) * 0.02).to(dt)
    one, zero, y = torch.ones(K, device="cuda"), torch.zeros(K, device="cuda"), torch.zeros(N, H, H, K, device="cuda", dtype=dt)
    d = sgs.ConvDesc(N=N, H=H, W=H, C=1 if depthwise else C, K=K, Kmax=K, Cmax=1 if depthwise else C, R=k, k=k, stride=1, act=1,
                     dtype=sgs.SGS_F32 if kind == "f32" else sgs.SGS_BF16, depthwise=int(depthwise))
    return x, y, lambda st: sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), one.data_ptr(), zero.data_ptr(), 0, y.data_ptr(), st)


def _linear(_):
    x, w, b = torch.randn(3, 512, device="cuda"), torch.randn(100, 512, device="cuda").bfloat16(), torch.zeros(100, device="cuda")
    y = torch.zeros(3, 100, device="cuda")
    d = sgs.AuxDesc(kind=SGS_AUX_LINEAR, dtype=sgs.SGS_BF16, N=3, H=1, W=1, C=512, K=100, ld=512)
    return x, y, lambda st: sgs.aux_op([d], [sgs.AuxArgs(x=x.data_ptr(), y=y.data_ptr(), w=w.data_ptr(), bias=b.data_ptr())], False, st)


def _query(kind):
    fam = {"resnet": wl.RESNET, "mbv3": wl.MBV3}[kind]
    net = gu.nets(fam, True)[2]
    x, y = torch.randn(2, 64, 64, 3, device="cuda").bfloat16(), torch.zeros(2, 1000, device="cuda")
    cfg = wl.extreme_cfg(fam, True)
    return x, y, lambda st: net.subnet_run(cfg, x.data_ptr(), 2, 64, y.data_ptr(), st)


@pytest.mark.parametrize("make,kind", [(_conv, "bf16"), (_conv, "f32"), (_conv, "depthwise"), (_linear, ""), (_query, "resnet"), (_query, "mbv3")])
def test_captured_calls_replay(make, kind):
    x, y, call = make(kind)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    call(st.cuda_stream)  # set-up: status word, shared-memory limits, workspaces, plans
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        call(st.cuda_stream)
        call(st.cuda_stream)  # (twice: a launch that starts under the one before, inside the graph)
    for seed in range(3):
        x.copy_(torch.randn(x.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed)))
        y.zero_()
        graph.replay()
        torch.cuda.synchronize()
        got = y.clone()
        y.zero_()
        torch.cuda.synchronize()
        call(st.cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(got, y) and y.abs().sum() > 0
    assert sgs.device_status() == 0


def test_a_query_is_captured_while_the_cached_subgraph_changes():
    # window 1: every query is a caching decision, so the capture begins with a table the device has not seen yet, and changes it
    net = sgs.SuperNet(wl.RESNET, gu.nets(wl.RESNET, True)[0], sgs.SGS_BF16)
    cfgs, res = wl.cfg_array([wl.extreme_cfg(wl.RESNET, False), wl.extreme_cfg(wl.RESNET, True)]), 64
    x, y = torch.randn(1, res, res, 3, device="cuda").bfloat16(), torch.zeros(2, 1000, device="cuda")
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    run = lambda i: net.subnet_run(cfgs[i], x.data_ptr(), 1, res, y[i].data_ptr(), st.cuda_stream)
    for i in (0, 1):
        run(i)
    torch.cuda.synchronize()
    want = y.clone()
    net.cache_configure(True, 0, 1)
    run(0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        run(1)
        run(0)
    assert net.cache_stats().decisions == 3
    y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    y.zero_()
    torch.cuda.synchronize()
    run(1)
    run(0)
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    net.close()


def test_grouped_layers_refuse_capture():
    x, y, b = torch.randn(3, 512, device="cuda"), torch.zeros(3, 100, device="cuda"), torch.zeros(100, device="cuda")
    w = torch.randn(100, 512, device="cuda").bfloat16()
    d = sgs.AuxDesc(kind=SGS_AUX_LINEAR, dtype=sgs.SGS_BF16, N=3, H=1, W=1, C=512, K=100, ld=512)
    st, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        with pytest.raises(sgs.SgsError) as e:
            sgs.aux_op([d], [sgs.AuxArgs(x=x.data_ptr(), y=y.data_ptr(), w=w.data_ptr(), bias=b.data_ptr())], True, st.cuda_stream)
        y.add_(1)  # (the capture itself goes on)
    assert e.value.status == SGS_EINVAL
    y.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert float(y.sum()) == y.numel()


@pytest.mark.parametrize("opts", [dict(wave=4, concurrency=2), dict(), dict(persistent=1)])
def test_streams_refuse_capture(opts):
    net = gu.nets(wl.MBV3, True)[2]
    n, res = 6, 64
    cfgs, x = wl.uniform_stream(wl.MBV3, n, seed=3), torch.randn(n, res, res, 3, device="cuda").bfloat16()
    y = torch.zeros(n, 1000, device="cuda")
    st = torch.cuda.Stream()
    run = lambda: net.stream_run(cfgs, x.data_ptr(), 1, res, y.data_ptr(), sgs.StreamOpts(cache_enabled=1, window_q=4, **opts), st.cuda_stream)
    torch.cuda.synchronize()
    run()
    want = y.cpu().numpy()
    other = torch.zeros(8, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        with pytest.raises(sgs.SgsError) as e:
            run()
        other.add_(1)  # (the capture itself goes on)
    assert e.value.status == SGS_EINVAL
    graph.replay()
    y.zero_()
    torch.cuda.synchronize()
    assert float(other[0]) == 1
    run()
    np.testing.assert_array_equal(y.cpu().numpy(), want)
