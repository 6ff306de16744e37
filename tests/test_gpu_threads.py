"""The layer entry points from several host threads, each on a stream of its own, among them every launcher's first use on the
device: what the threads share (shared-memory limits, device facts) is set while others read it."""
import subprocess
import sys

import pytest
import torch

pytestmark = pytest.mark.gpu

PROGRAM = r"""
import threading
import torch
import paper_2306_17266_b200 as sgs

def layer(N, H, C, K, k, dtype, depthwise, stream, y):
    g = torch.Generator(device="cuda").manual_seed(K + k)
    x = torch.randn(N, H, H, C, device="cuda", generator=g).to(dtype)
    w = (torch.randn(k, k, K, device="cuda", generator=g) if depthwise else torch.randn(K, k, k, C, device="cuda", generator=g) * 0.05).to(dtype)
    one, zero = torch.ones(K, device="cuda"), torch.zeros(K, device="cuda")
    d = sgs.ConvDesc(N=N, H=H, W=H, C=1 if depthwise else C, K=K, Kmax=K, Cmax=1 if depthwise else C, R=k, k=k, stride=1, act=1,
                     dtype=sgs.SGS_BF16 if dtype == torch.bfloat16 else sgs.SGS_F32, depthwise=int(depthwise))
    torch.cuda.synchronize()
    return (x, w, one, zero), lambda: sgs.conv2d_sliced(d, x.data_ptr(), w.data_ptr(), one.data_ptr(), zero.data_ptr(), 0, y.data_ptr(), stream.cuda_stream)

# fp32 tiles above 48 KB, depthwise rings above 47 KB (5x5 and 7x7, wide and narrow maps), tensor cores
LAYERS = [(2, 40, 64, 128, 3, torch.float32, False), (1, 9, 128, 64, 1, torch.float32, False), (1, 30, 64, 64, 5, torch.bfloat16, True),
          (1, 30, 64, 64, 7, torch.bfloat16, True), (1, 9, 64, 64, 7, torch.bfloat16, True), (1, 14, 64, 128, 3, torch.bfloat16, False)]
THREADS, ROUNDS = 4, 20
work = []
for t in range(THREADS):
    stream = torch.cuda.Stream()
    for l in LAYERS:
        y = torch.zeros(l[0], l[1], l[1], l[3], device="cuda", dtype=l[5])
        work.append((t, y, *layer(*l, stream, y)))
start, errors = threading.Barrier(THREADS), []

def serve(t):
    try:
        start.wait()
        for r in range(ROUNDS):
            mine = [w[3] for w in work if w[0] == t]
            for call in mine[t % len(mine):] + mine[:t % len(mine)]:  # (the threads begin with different layers)
                call()
    except Exception as e:
        errors.append(e)

threads = [threading.Thread(target=serve, args=(t,)) for t in range(THREADS)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not errors, errors
n = len(LAYERS)
for i in range(n):
    first = work[i][1]
    assert first.abs().sum() > 0
    for t in range(1, THREADS):
        assert torch.equal(first, work[t * n + i][1]), (i, t)
assert sgs.device_status() == 0
print("ok")
"""


def test_first_use_from_several_threads():
    assert torch.cuda.is_available()
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-2000:] + r.stderr[-2000:]
