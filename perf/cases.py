"""Workloads on which the library's speed is measured, through its public entry points.

``listed()`` names the fixed ones, ``draw(rng)`` gives another of the same ranges; ``prepare`` makes what a program has in
hand before the call (a loaded SuperNet, device or pinned host buffers, the array of SubNet configs), ``run`` is one pass.

Kinds of a case:
  query   one SubNet on a batch of images: sgs_subnet_run                     (family, dtype, batch, res, cfg_seed)
  stream  a stream of queries, each with its own SubNet: sgs_stream_run, or sgs_stream_run_host with host buffers
          (family, n, batch, res, locality, mode, wave, in_flight, host, cfg_seed)
  dw      one depthwise layer with its folded batch norm and activation       (N, H, W, K, k, stride, act)
  i8      one sliced 8-bit convolution layer                                  (N, H, W, C, K, k, stride, residual)
"""
import math

import numpy as np
import torch

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl

FAMILY = {"tiny": wl.TINY, "resnet": wl.RESNET, "mbv3": wl.MBV3}
DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}


def query(family, dtype, batch, res, cfg_seed):
    return {"kind": "query", "family": family, "dtype": dtype, "batch": batch, "res": res, "cfg_seed": cfg_seed}


def stream(family, n, batch, res, mode, wave=0, in_flight=1, locality=False, host=False, cfg_seed=2):
    return {"kind": "stream", "family": family, "n": n, "batch": batch, "res": res, "mode": mode, "wave": wave, "in_flight": in_flight,
            "locality": locality, "host": host, "cfg_seed": cfg_seed}


def dw(N, H, W, K, k, stride, act):
    return {"kind": "dw", "N": N, "H": H, "W": W, "K": K, "k": k, "stride": stride, "act": act}


def i8(N, H, W, C, K, k, stride, residual):
    return {"kind": "i8", "N": N, "H": H, "W": W, "C": C, "K": K, "k": k, "stride": stride, "residual": residual}


def listed():
    return [
        # the smallest call: one 32x32 image through a SubNet of the tiny SuperNet in fp32; launches are all it costs
        dict(query("tiny", "f32", 1, 32, 0), name="tiny_query_f32"),
        # one query at a time, as a latency-bound server issues them: the two SuperNets of the paper, one image
        dict(query("resnet", "bf16", 1, 224, 2), name="resnet_query"),
        dict(query("mbv3", "bf16", 1, 224, 3), name="mbv3_query"),
        # the full-precision mode, on a small batch at a reduced resolution
        dict(query("resnet", "f32", 3, 160, 5), name="resnet_query_f32"),
        # the benchmark's stream: uniform SubNets, one image each, waves of 32 with four in flight
        dict(stream("resnet", 128, 1, 224, "wave", 32, 4), name="resnet_stream"),
        # the same from pinned host buffers, with a ragged last wave, at another resolution
        dict(stream("resnet", 75, 1, 192, "wave", 32, 4, host=True, cfg_seed=7), name="resnet_stream_host"),
        # the throughput sweep: 16 images per query, waves of four configs
        dict(stream("resnet", 48, 16, 224, "wave", 4, 4, cfg_seed=4), name="resnet_sweep_b16"),
        # the locality stream at batch 16, served one query at a time with the SubGraph cache on
        dict(stream("resnet", 8, 16, 224, "one", locality=True, cfg_seed=4), name="resnet_locality_b16"),
        # the depthwise-heavy family: in waves, and as one launch of the persistent kernel (more queries than SMs, last round ragged)
        dict(stream("mbv3", 96, 1, 224, "wave", 32, 4, cfg_seed=3), name="mbv3_stream"),
        dict(stream("mbv3", 333, 1, 224, "persistent", cfg_seed=3), name="mbv3_persistent"),
        # one large depthwise layer (the middle kernel size), beyond L2
        dict(dw(64, 56, 56, 480, 5, 1, 2), name="depthwise_k5"),
        # the paper's 8-bit format, a 3x3 layer in the middle of the network at batch 16
        dict(i8(16, 28, 28, 176, 176, 3, 1, False), name="int8_conv3x3"),
    ]


def _log(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    seed = rng.randrange(1 << 20)
    what = rng.choices(["query", "wave", "one", "persistent", "dw", "i8"], [4, 4, 1, 1, 1, 1])[0]
    res = 16 * rng.randint(8, 15)  # 128 .. 240, not only the multiples of the networks' total stride
    if what == "query":
        family = rng.choice(["tiny", "resnet", "resnet", "mbv3"])
        if family == "tiny":
            return query("tiny", rng.choice(["f32", "bf16"]), _log(rng, 1, 32), 8 * rng.randint(3, 8), seed)
        if rng.random() < 0.25:
            return query(family, "f32", _log(rng, 1, 4), min(res, 192), seed)
        return query(family, "bf16", _log(rng, 1, 16), res, seed)
    if what == "wave":
        if rng.random() < 0.3:  # several images per query, few queries per wave
            batch = _log(rng, 2, 16)
            n = _log(rng, 4, max(4, 512 // batch))
            return stream("resnet", n, batch, min(res, 224), "wave", 4, rng.randint(2, 4), rng.random() < 0.5, rng.random() < 0.25, seed)
        family = rng.choice(["resnet", "mbv3"])
        return stream(family, _log(rng, 5, 256), 1, res, "wave", rng.choice([8, 16, 32]), rng.randint(1, 4), rng.random() < 0.5,
                      rng.random() < 0.25, seed)
    if what == "one":
        batch = _log(rng, 1, 16)
        return stream(rng.choice(["resnet", "mbv3"]), _log(rng, 2, max(2, 64 // batch)), batch, min(res, 224), "one", locality=True, cfg_seed=seed)
    if what == "persistent":
        return stream("mbv3", _log(rng, 2, 600), 1, min(res, 224), "persistent", locality=rng.random() < 0.5, host=rng.random() < 0.25, cfg_seed=seed)
    if what == "dw":
        H = rng.choice([7, 14, 20, 28, 35, 56, 75, 112])
        K = 8 * _log(rng, 2, 120)
        N = _log(rng, 1, max(1, min(256, 90_000_000 // (H * H * K))))
        return dw(N, H, H, K, rng.choice([3, 5, 7]), rng.choice([1, 2]), rng.choice([1, 2]))
    H = rng.choice([7, 14, 28, 56])
    stride = rng.choice([1, 2]) if H % 2 == 0 else 1
    C = 16 * _log(rng, 2, 2048 // (4 * H))
    k = rng.choice([1, 3])
    K = 8 * _log(rng, 4, 2 * 2048 // (4 * H)) if k == 3 else 8 * _log(rng, 4, 8 * 2048 // (4 * H))
    return i8(_log(rng, 1, 32), H, H, C, K, k, stride, rng.random() < 0.3)


# A program loads its SuperNet once and serves everything from it on one stream (a handle takes one stream at a time): both
# live as long as the process.
_nets = {}
_streams = []


def _stream():
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def _net(family, dtype):
    key = (family, dtype)
    if key not in _nets:
        blob = wl.make_blob(FAMILY[family], seed=0, bf16_weights=dtype == "bf16")
        _nets[key] = sgs.SuperNet(FAMILY[family], blob, sgs.SGS_BF16 if dtype == "bf16" else sgs.SGS_F32)
    return _nets[key]


def _configs(case):
    family = FAMILY[case["family"]]
    if case["kind"] == "query":
        return wl.uniform_stream(family, 1, case["cfg_seed"])
    if case["locality"]:
        return wl.markov_stream(case["n"], case["cfg_seed"], family=family)
    return wl.uniform_stream(family, case["n"], case["cfg_seed"])


def _out(size, k, stride):
    return (size + 2 * ((k - 1) // 2) - k) // stride + 1


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case, "stream": _stream()}
    if case["kind"] in ("query", "stream"):
        dtype = case.get("dtype", "bf16")
        net = s["net"] = _net(case["family"], dtype)
        n = case.get("n", 1) * case["batch"]
        s["x"] = torch.randn(n, case["res"], case["res"], 3, device="cuda", generator=g).to(DTYPE[dtype])
        s["logits"] = torch.zeros(n, net.n_classes, device="cuda")
        s["cfgs"] = wl.cfg_array(_configs(case))
        if case["kind"] == "stream":
            if case["host"]:
                s["x"], s["logits"] = s["x"].cpu().pin_memory(), s["logits"].cpu().pin_memory()
            one = case["mode"] == "one"
            s["opts"] = sgs.StreamOpts(cache_enabled=1, window_q=4, cache_budget_bytes=0, use_graphs=1, record_latency=int(one),
                                       concurrency=case["in_flight"], wave=case["wave"], persistent=int(case["mode"] == "persistent"))
    elif case["kind"] == "dw":
        N, H, W, K, k, stride = (case[v] for v in ("N", "H", "W", "K", "k", "stride"))
        # what a depthwise layer meets: the output of the expansion's activation
        s["x"] = torch.nn.functional.hardswish(torch.randn(N, H, W, K, device="cuda", generator=g, dtype=torch.bfloat16))
        s["w"] = (torch.randn(7, 7, K, device="cuda", generator=g) * (2 / 49) ** 0.5).to(torch.bfloat16)
        s["scale"] = torch.rand(K, device="cuda", generator=g) + 0.5
        s["shift"] = torch.randn(K, device="cuda", generator=g) * 0.1
        s["y"] = torch.empty(N, _out(H, k, stride), _out(W, k, stride), K, device="cuda", dtype=torch.bfloat16)
        s["desc"] = sgs.ConvDesc(N=N, H=H, W=W, C=1, K=K, Kmax=K, Cmax=1, R=7, k=k, stride=stride, act=case["act"], dtype=sgs.SGS_BF16,
                                 depthwise=1)
    else:
        N, H, W, C, K, k, stride = (case[v] for v in ("N", "H", "W", "C", "K", "k", "stride"))
        Cmax, Kmax = C + 16, K + 16  # a slice of a slightly larger stored layer
        shape = (N, _out(H, k, stride), _out(W, k, stride), K)
        s["x"] = torch.randint(0, 256, (N, H, W, C), device="cuda", generator=g, dtype=torch.uint8)
        s["w"] = torch.randint(-127, 128, (Kmax, k, k, Cmax), device="cuda", generator=g, dtype=torch.int8)
        # multipliers that bring the accumulator (up to ~ 255 * 127 * C * k * k / 3) into the byte range
        real = (96.0 / (128 * 64 * math.sqrt(C * k * k))) * (torch.rand(Kmax, device="cuda", generator=g, dtype=torch.float64) + 0.5)
        shift = torch.clamp(torch.floor(-torch.log2(real)), 0, 31)
        s["mult"] = torch.clamp(torch.round(real * 2.0 ** (31 + shift)), max=2.0 ** 31 - 1).to(torch.int32)
        s["shift"] = shift.to(torch.int32)
        s["bias"] = torch.randint(-30, 30, (Kmax,), device="cuda", generator=g, dtype=torch.int32)
        s["res"] = torch.randint(0, 256, shape, device="cuda", generator=g, dtype=torch.uint8) if case["residual"] else None
        s["y"] = torch.empty(shape, device="cuda", dtype=torch.uint8)
        s["desc"] = sgs.ConvI8Desc(N=N, H=H, W=W, C=C, K=K, Kmax=Kmax, Cmax=Cmax, R=k, k=k, stride=stride, relu=1, zy=7, zr=11,
                                   res_mult=1932735283, res_shift=1)
    return s


def run(s):
    case, st = s["case"], s["stream"].cuda_stream
    if case["kind"] == "query":
        s["net"].subnet_run(s["cfgs"][0], s["x"].data_ptr(), case["batch"], case["res"], s["logits"].data_ptr(), st)
        return s["logits"]
    if case["kind"] == "stream":
        stats = s["net"].stream_run(s["cfgs"], s["x"].data_ptr(), case["batch"], case["res"], s["logits"].data_ptr(), s["opts"], st,
                                    host=case["host"])
        return {"logits": s["logits"], "hbm_weight_bytes": stats.hbm_weight_bytes, "hit_ratio": stats.hit_ratio,
                "weight_bytes": stats.weight_bytes, "useful_flops": stats.useful_flops}
    if case["kind"] == "dw":
        sgs.conv2d_sliced(s["desc"], s["x"].data_ptr(), s["w"].data_ptr(), s["scale"].data_ptr(), s["shift"].data_ptr(), 0,
                          s["y"].data_ptr(), st)
        return s["y"]
    sgs.conv2d_sliced_i8(s["desc"], s["x"].data_ptr(), s["w"].data_ptr(), s["mult"].data_ptr(), s["shift"].data_ptr(), s["bias"].data_ptr(),
                         s["res"].data_ptr() if s["res"] is not None else 0, s["y"].data_ptr(), st)
    return s["y"]


def _union(boxes):
    """Elements of the union of prefix boxes (K filters x n elements of each)."""
    total, reach = 0, 0
    for K, n in sorted(boxes, reverse=True):  # widest prefix first: a narrower one adds only what lies beyond `reach`
        if n > reach:
            total += K * (n - reach)
            reach = n
    return total


def work(case):
    """Images and the weights that the SubNets of the call use, each once, and the logits; the SubNets' useful operations."""
    if case["kind"] in ("query", "stream"):
        dtype = case.get("dtype", "bf16")
        net, elem = _net(case["family"], dtype), 2 if dtype == "bf16" else 4
        boxes, flops, known = [set() for _ in range(net.n_layers)], 0.0, {}
        for c in _configs(case):
            if c.key() not in known:
                known[c.key()] = net.subnet_cost(c, case["batch"], case["res"])[0]
                for i, (K, C, k) in enumerate(net.subnet_encode(c).tolist()):
                    boxes[i].add((K, C * k * k))
            flops += known[c.key()]
        n = case.get("n", 1) * case["batch"]
        nbytes = n * (case["res"] ** 2 * 3 * elem + net.n_classes * 4) + elem * sum(_union(b) for b in boxes)
        return {"bytes": nbytes, "flops": flops}
    N, H, W, K, k, stride = (case[v] for v in ("N", "H", "W", "K", "k", "stride"))
    M = N * _out(H, k, stride) * _out(W, k, stride)
    if case["kind"] == "dw":
        return {"bytes": 2 * (N * H * W * K + M * K + k * k * K) + 8 * K, "flops": 2.0 * M * K * k * k}
    C = case["C"]
    return {"bytes": N * H * W * C + M * K * (2 if case["residual"] else 1) + K * C * k * k + 12 * K, "flops": 2.0 * M * K * C * k * k}


def tolerance(case):
    if case["kind"] == "i8":
        return "exact"  # whole-number arithmetic
    if case["kind"] == "dw":
        return {"rel": 5e-3, "max": 2e-2}  # fp32 sums of bf16 products, stored as bf16: an output is off by one rounding step at most
    if case.get("dtype") == "f32":
        return {"rel": 1e-5, "max": 1e-4}  # 32-bit sums, up to some 60 layers deep
    return {"rel": 1e-2, "max": 1e-1}  # every layer's output rounded to bf16: a few steps differ with the order of the sums
