"""Weights and parameters that the previous kernel of the stream writes.  The layer entry points start a kernel before the one
ahead of it has finished; what the caller hands over, weights included, may come from that kernel.  Every layer runs in a
chain in which each call's weights are the output of the call before it, enqueued without a pause, and has to give exactly
what it gives with a synchronisation after every call."""
import pytest
import torch

import paper_2306_17266_b200 as sgs

pytestmark = pytest.mark.gpu

ROUNDS = 12


def _rand(*shape, seed):
    return torch.randn(*shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


def _conv(x, w, scale, shift, y, *, depthwise=False, impl=0):
    """x [N][H][W][C], y [N][H][W][K], stride 1, no activation; w [K][k][k][C], depthwise [k][k][K]."""
    N, H, W, C = x.shape
    K, k = (w.shape[2], w.shape[0]) if depthwise else (w.shape[0], w.shape[1])
    d = sgs.ConvDesc(N=N, H=H, W=W, C=1 if depthwise else C, K=K, Kmax=K, Cmax=1 if depthwise else C, R=k, k=k, stride=1, act=0, impl=impl,
                     dtype=sgs.SGS_BF16 if x.dtype == torch.bfloat16 else sgs.SGS_F32, depthwise=int(depthwise))
    sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), scale.data_ptr(), shift.data_ptr(), 0, y.data_ptr(), torch.cuda.current_stream().cuda_stream)


def _check(produce, consume, make_out):
    """produce(i) writes the weights of round i, consume(y) uses them."""
    outs = {}
    for wait in (True, False):
        outs[wait] = [make_out() for _ in range(ROUNDS)]
        torch.cuda.synchronize()
        for i, y in enumerate(outs[wait]):
            produce(i)
            if wait:
                torch.cuda.synchronize()
            consume(y)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        assert sgs.device_status() == 0
    assert not torch.equal(outs[True][0], outs[True][1])  # (the rounds differ)
    for a, b in zip(outs[True], outs[False]):
        assert torch.equal(a, b)


def _matrix_producer(rows, cols, dtype, impl=0):
    """A [rows][cols] tensor written by a matrix product of the library, another one in every round."""
    w = torch.zeros(rows, cols, device="cuda", dtype=dtype)
    xs = [_rand(1, 1, rows, 512, seed=i).to(dtype) for i in range(ROUNDS)]
    b = (_rand(cols, 1, 1, 512, seed=99) * 0.02).to(dtype)
    one, zero = torch.ones(cols, device="cuda"), torch.zeros(cols, device="cuda")
    return w, lambda i: _conv(xs[i], b, one, zero, w.view(1, 1, rows, cols), impl=impl)


@pytest.mark.parametrize("N,H,C,K,k", [(1, 7, 512, 1024, 1), (1, 7, 64, 128, 3), (8, 28, 64, 256, 1)])
def test_tensor_core_weights(N, H, C, K, k):
    w, produce = _matrix_producer(K * k * k, C, torch.bfloat16)
    x, one, zero = _rand(N, H, H, C, seed=5).bfloat16(), torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    _check(produce, lambda y: _conv(x, w.view(K, k, k, C), one, zero, y, impl=2), lambda: torch.zeros(N, H, H, K, device="cuda", dtype=torch.bfloat16))


def test_static_entry_point_weights():
    K, C, H = 1024, 512, 7
    w, produce = _matrix_producer(K, C, torch.bfloat16)
    x, one, zero = _rand(1, H, H, C, seed=5).bfloat16(), torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    d = sgs.ConvDesc(N=1, H=H, W=H, C=C, K=K, Kmax=K, Cmax=C, R=1, k=1, stride=1, act=0, dtype=sgs.SGS_BF16, split_k_off=1)

    def consume(y):
        sgs.conv2d_sliced_static(d, x.data_ptr(), w.data_ptr(), one.data_ptr(), zero.data_ptr(), 0, y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    _check(produce, consume, lambda: torch.zeros(1, H, H, K, device="cuda", dtype=torch.bfloat16))


@pytest.mark.parametrize("which", ["scale", "shift"])
def test_folded_batch_norm(which):
    # the parameters are one row of a fully connected layer's output
    K, C, H = 512, 256, 14
    par = {"scale": torch.ones(K, device="cuda"), "shift": torch.zeros(K, device="cuda")}
    wl, bl = (_rand(K, 1024, seed=7) * 0.05).bfloat16(), torch.zeros(K, device="cuda")
    vs = [_rand(1, 1024, seed=20 + i) for i in range(ROUNDS)]
    d = sgs.AuxDesc(kind=sgs.binding.SGS_AUX_LINEAR, dtype=sgs.SGS_BF16, N=1, H=1, W=1, C=1024, K=K, ld=1024, act=0)

    def produce(i):
        sgs.aux_op([d], [sgs.AuxArgs(x=vs[i].data_ptr(), y=par[which].data_ptr(), w=wl.data_ptr(), bias=bl.data_ptr())], False,
                   torch.cuda.current_stream().cuda_stream)
    x, w = _rand(1, H, H, C, seed=3).bfloat16(), (_rand(K, 1, 1, C, seed=4) * 0.06).bfloat16()
    _check(produce, lambda y: _conv(x, w, par["scale"], par["shift"], y, impl=2), lambda: torch.zeros(1, H, H, K, device="cuda", dtype=torch.bfloat16))


def test_int8_weights():
    # weights = the bytes another 8-bit layer wrote
    K, C, H = 512, 256, 14
    w = torch.zeros(K, C, device="cuda", dtype=torch.uint8)
    g = torch.Generator(device="cuda").manual_seed(1)
    xs = [torch.randint(0, 256, (1, 1, K, 512), device="cuda", generator=g, dtype=torch.uint8) for _ in range(ROUNDS)]
    b = torch.randint(-127, 128, (C, 1, 1, 512), device="cuda", generator=g, dtype=torch.int8)
    x = torch.randint(0, 256, (1, H, H, C), device="cuda", generator=g, dtype=torch.uint8)

    def layer(x, w, y, K, C, N, H, W, y_signed):
        mult, shift, bias = (torch.full((K,), v, device="cuda", dtype=torch.int32) for v in (2 ** 30, 12, 3))
        d = sgs.ConvI8Desc(N=N, H=H, W=W, C=C, K=K, Kmax=K, Cmax=C, R=1, k=1, stride=1, relu=0, y_signed=y_signed)
        return lambda xi, yi: sgs.conv2d_sliced_i8(d, xi.data_ptr(), w.data_ptr(), mult.data_ptr(), shift.data_ptr(), bias.data_ptr(), 0, yi.data_ptr(),
                                                   torch.cuda.current_stream().cuda_stream)
    first, second = layer(xs[0], b, w, C, 512, 1, 1, K, 1), layer(x, w, None, K, C, 1, H, H, 0)
    _check(lambda i: first(xs[i], w), lambda y: second(x, y), lambda: torch.zeros(1, H, H, K, device="cuda", dtype=torch.uint8))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_cuda_core_weights(dtype):
    K, C, H = 256, 128, 9
    w, produce = _matrix_producer(K, C, dtype, impl=1)
    x, one, zero = _rand(1, H, H, C, seed=5).to(dtype), torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    _check(produce, lambda y: _conv(x, w.view(K, 1, 1, C), one, zero, y, impl=1), lambda: torch.zeros(1, H, H, K, device="cuda", dtype=dtype))


def test_depthwise_weights():
    K, H = 512, 14
    w, produce = _matrix_producer(25, K, torch.bfloat16)
    x, one, zero = _rand(2, H, H, K, seed=5).bfloat16(), torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    _check(produce, lambda y: _conv(x, w.view(5, 5, K), one, zero, y, depthwise=True), lambda: torch.zeros(2, H, H, K, device="cuda", dtype=torch.bfloat16))


# (rows, inputs): one and many rows of the vectorised kernel, the scalar kernel
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("N,C", [(1, 512), (16, 512), (2, 508)])
def test_linear_weights(N, C, dtype):
    K = 1024
    w, produce = _matrix_producer(K, 512, dtype, impl=0 if dtype == torch.bfloat16 else 1)
    v, b = _rand(N, C, seed=5), torch.zeros(K, device="cuda")
    d = sgs.AuxDesc(kind=sgs.binding.SGS_AUX_LINEAR, dtype=sgs.SGS_BF16 if dtype == torch.bfloat16 else sgs.SGS_F32, N=N, H=1, W=1, C=C, K=K, ld=512, act=0)
    _check(produce, lambda y: sgs.aux_op([d], [sgs.AuxArgs(x=v.data_ptr(), y=y.data_ptr(), w=w.data_ptr(), bias=b.data_ptr())], False,
                                         torch.cuda.current_stream().cuda_stream), lambda: torch.zeros(N, K, device="cuda"))


def test_squeeze_excite_gate_weights():
    mid, sq = 480, 120
    w1, produce = _matrix_producer(sq, mid, torch.bfloat16)
    w2, g = (_rand(mid, sq, seed=6) * 0.1).bfloat16(), _rand(3, mid, seed=7)
    b1, b2 = torch.zeros(sq, device="cuda"), torch.zeros(mid, device="cuda")
    d = sgs.AuxDesc(kind=sgs.binding.SGS_AUX_SE_GATE, dtype=sgs.SGS_BF16, N=3, H=1, W=1, C=mid, K=sq, ld=mid, ld2=sq)
    _check(produce, lambda y: sgs.aux_op([d], [sgs.AuxArgs(x=g.data_ptr(), y=y.data_ptr(), w=w1.data_ptr(), bias=b1.data_ptr(), w2=w2.data_ptr(),
                                                           bias2=b2.data_ptr())], False, torch.cuda.current_stream().cuda_stream),
           lambda: torch.zeros(3, mid, device="cuda"))
