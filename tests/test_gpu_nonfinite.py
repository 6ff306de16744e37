"""NaN and infinities through the epilogues: a layer without activation passes them on, ReLU makes a NaN zero (its maximum), on
the tensor-core, CUDA-core, depthwise, grouped and persistent kernels alike."""
import numpy as np
import pytest
import torch

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# impl 2 with whole tiles, with reductions split over 2 .. 8 blocks, with a residual; impl 1; depthwise strips of 4 and 8 columns
@pytest.mark.parametrize("act", [0, 1])
@pytest.mark.parametrize("impl,N,H,C,K,k,residual", [(2, 16, 28, 64, 152, 1, False), (2, 1, 7, 1024, 72, 1, True), (2, 1, 14, 512, 256, 3, False),
                                                     (1, 1, 9, 40, 24, 3, True), (0, 1, 9, 72, 72, 5, False), (0, 1, 30, 72, 72, 3, False)])
def test_layer_epilogues(impl, N, H, C, K, k, residual, act):
    g = torch.Generator(device="cuda").manual_seed(2)
    depthwise = impl == 0
    x = torch.randn(N, H, H, C, device="cuda", generator=g).bfloat16()
    x[0, 0, 1, 3], x[0, H - 1, H - 2, 5], x[0, H // 2, 0, 7] = float("nan"), float("inf"), -float("inf")
    w = (torch.randn(k, k, K, device="cuda", generator=g) if depthwise else torch.randn(K, k, k, C, device="cuda", generator=g) / (C * k * k) ** 0.5).bfloat16()
    one, zero = torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    res = torch.randn(N, H, H, K, device="cuda", generator=g).bfloat16() if residual else None
    y = torch.zeros(N, H, H, K, device="cuda", dtype=torch.bfloat16)
    d = sgs.ConvDesc(N=N, H=H, W=H, C=1 if depthwise else C, K=K, Kmax=K, Cmax=1 if depthwise else C, R=k, k=k, stride=1, act=act, dtype=sgs.SGS_BF16,
                     impl=impl, depthwise=int(depthwise))
    sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), one.data_ptr(), zero.data_ptr(), res.data_ptr() if residual else 0, y.data_ptr(),
                      torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    wt = w.permute(2, 0, 1).unsqueeze(1) if depthwise else w.permute(0, 3, 1, 2)
    ref = torch.nn.functional.conv2d(x.cpu().double().permute(0, 3, 1, 2), wt.cpu().double(), padding=k // 2, groups=K if depthwise else 1).permute(0, 2, 3, 1)
    ref = ref + res.cpu().double() if residual else ref
    if act == 1:
        ref = torch.where(ref > 0, ref, torch.zeros_like(ref))
    got = y.cpu().double()
    assert torch.isnan(ref).any() == (act == 0) and torch.isinf(ref).any()
    assert torch.equal(torch.isnan(got), torch.isnan(ref))
    assert torch.equal(torch.isinf(got), torch.isinf(ref)) and torch.equal(got[torch.isinf(ref)], ref[torch.isinf(ref)])
    fin = torch.isfinite(ref)
    assert (got[fin] - ref[fin]).abs().max() <= 1e-2 * ref[fin].abs().max()


def test_nan_parameter_of_a_linear_bottleneck_in_every_execution():
    # One filter of a layer without activation has a NaN shift; the ReLU of the next layer turns what it touches into zeros, so
    # the logits are finite, and the same whatever executes the SubNet.
    blob = wl.make_blob(wl.MBV3, seed=0, bf16_weights=True)
    words, pos = blob.view(np.float32), 8
    for r in wl.supernet_records(wl.MBV3):
        pos += 8
        if r.name == "s0b0.project":
            words[pos + r.n_weights + r.K + 5] = np.nan  # beta of filter 5 (gamma, beta, mean, var follow the weights)
        pos += r.n_floats
    net = sgs.SuperNet(wl.MBV3, blob, sgs.SGS_BF16)
    n, res = 6, 64
    cfgs = wl.uniform_stream(wl.MBV3, n, seed=3)
    x = gu.to_device(wl.make_inputs(n, 1, res, seed=1, bf16=True).reshape(n, res, res, 3), True)
    st = torch.cuda.Stream()

    def stream_run(**opts):
        y = torch.zeros(n, net.n_classes, device="cuda")
        torch.cuda.synchronize()
        net.stream_run(cfgs, x.data_ptr(), 1, res, y.data_ptr(), sgs.StreamOpts(cache_enabled=1, window_q=4, **opts), st.cuda_stream)
        return y.cpu().numpy()
    runs = {"waves": stream_run(wave=4, concurrency=2), "one by one": stream_run(), "persistent": stream_run(persistent=1)}
    net.set_option("conv_impl", 1)
    ref = stream_run()
    net.close()
    assert np.isfinite(ref).all()
    for name, y in runs.items():
        assert np.isfinite(y).all(), name
        assert gu.rel_err(y, ref) <= 2e-2, name
