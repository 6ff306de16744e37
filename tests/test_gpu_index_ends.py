"""Layers so large that an element, output or thread index is about to leave its 32 bits."""
import pytest
import torch

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200.binding import SGS_AUX_AVGPOOL, SGS_AUX_LINEAR, SGS_AUX_SE_SCALE

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _memory():
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 48 << 30:
        pytest.skip("needs 48 GB of free device memory")
    yield
    torch.cuda.empty_cache()


def _run(desc, args, grouped):
    sgs.aux_op([desc], [args], grouped, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()


def test_scale_of_almost_two_to_the_31_vectors():
    # the grid-stride loop's last step ends past 2^31 vectors of 8 channels
    N, H, C = (1 << 31) // (256 * 4) - 1, 256, 32
    x = torch.full((N, H, 1, C), 2.0, device="cuda", dtype=torch.bfloat16)
    gate = torch.rand(N, C, device="cuda")
    _run(sgs.AuxDesc(kind=SGS_AUX_SE_SCALE, dtype=sgs.SGS_BF16, N=N, H=H, W=1, C=C),
         sgs.AuxArgs(x=x.data_ptr(), y=x.data_ptr(), w=gate.data_ptr()), True)
    want = (2 * gate).bfloat16()
    for n0 in range(0, N, 1 << 17):
        part = x[n0:n0 + (1 << 17), :, 0]
        assert torch.equal(part, want[n0:n0 + (1 << 17), None].expand_as(part)), n0


@pytest.mark.parametrize("dtype,C", [(torch.bfloat16, 8), (torch.float32, 1)])
def test_linear_of_two_to_the_27_outputs(dtype, C):
    K = (1 << 27) + 64  # a warp per output: from 2^32 threads on
    w = torch.zeros(K, C, device="cuda", dtype=dtype)
    w[:, 0] = (torch.arange(K, device="cuda") % 251).to(dtype)
    x, bias, y = torch.full((1, C), 3.0, device="cuda"), torch.zeros(K, device="cuda"), torch.full((K,), -1.0, device="cuda")
    _run(sgs.AuxDesc(kind=SGS_AUX_LINEAR, dtype=sgs.SGS_BF16 if dtype == torch.bfloat16 else sgs.SGS_F32, N=1, H=1, W=1, C=C, K=K, ld=C),
         sgs.AuxArgs(x=x.data_ptr(), y=y.data_ptr(), w=w.data_ptr(), bias=bias.data_ptr()), False)
    assert torch.equal(y, 3 * w[:, 0].float())


@pytest.mark.parametrize("grouped", [False, True])
def test_average_pool_of_two_to_the_26_vectors(grouped):
    N, C = (1 << 20) + 3, 512
    x = (torch.arange(N * 2, device="cuda") % 127).to(torch.bfloat16).view(N, 2, 1, 1).expand(N, 2, 1, C).contiguous()
    y = torch.full((N, C), -1.0, device="cuda")
    _run(sgs.AuxDesc(kind=SGS_AUX_AVGPOOL, dtype=sgs.SGS_BF16, N=N, H=2, W=1, C=C), sgs.AuxArgs(x=x.data_ptr(), y=y.data_ptr()), grouped)
    want = x[:, :, 0, 0].float().mean(1)
    assert torch.equal(y, want[:, None].expand(N, C))


def test_linear_of_more_rows_than_one_grid_numbers():
    # two members of 300 000 images each: 75 000 groups of rows
    N, C, K = 300_000, 8, 10
    w, bias = torch.randn(K, C, device="cuda").bfloat16(), torch.randn(K, device="cuda")
    xs = [torch.randn(N, C, device="cuda") for _ in range(2)]
    ys = [torch.full((N, K), 77.0, device="cuda") for _ in range(2)]
    d = sgs.AuxDesc(kind=SGS_AUX_LINEAR, dtype=sgs.SGS_BF16, N=N, H=1, W=1, C=C, K=K, ld=C)
    sgs.aux_op([d, d], [sgs.AuxArgs(x=x.data_ptr(), y=y.data_ptr(), w=w.data_ptr(), bias=bias.data_ptr()) for x, y in zip(xs, ys)], True,
               torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for x, y in zip(xs, ys):
        ref = x.double() @ w.double().T + bias.double()
        assert (y.double() - ref).abs().max() <= 1e-6 * ref.abs().max()  # (fp32 sums of 8 terms)
