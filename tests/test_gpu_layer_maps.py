"""Output maps of single layers, where they lie in the network, element by element: the fused stem, the grouped kernel (waves, and the
large layers of a single query) and the latency kernel with its pairs.  The reference is a double-precision convolution of the map that
the layer in front left behind, so every element has to agree up to its own rounding."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu
from tests import torch_ref

pytestmark = pytest.mark.gpu

_params = {}


def params(fam):
    if fam not in _params:
        P = torch_ref.parse_blob(fam, gu.nets(fam, True)[0])
        _params[fam] = {k: {n: t.cuda() for n, t in d.items()} for k, d in P.items()}
    return _params[fam]


def run(gnet, cfgs, x, batch, res, wave):
    """One pass: single queries one after the other (wave 0: the last one's maps stay), or one wave."""
    stream = torch.cuda.Stream()
    out = torch.zeros(len(cfgs) * batch, gnet.n_classes, device="cuda")
    torch.cuda.synchronize()
    if wave:
        opts = sgs.StreamOpts(cache_enabled=1, window_q=4, record_latency=0, concurrency=1, wave=len(cfgs))
        gnet.stream_run(cfgs, x.data_ptr(), batch, res, out.data_ptr(), opts, stream.cuda_stream)
    else:
        gnet.subnet_run(wl.cfg_array(cfgs)[0], x.data_ptr(), batch, res, out.data_ptr(), stream.cuda_stream)
    torch.cuda.synchronize()


def maps_of(gnet, names, layer, cfgs, x, batch, res, wave):
    """Per member: the map of stored layer `layer` [N][H][W][K] (None where its SubNet does not use it); its padding has to be zero."""
    li = names.index(layer)
    buf = torch.full((min(batch * res * res * 384 + (1 << 16), 1 << 31),), float("nan"), dtype=torch.bfloat16, device="cuda")
    arr = wl.cfg_array(cfgs)
    gnet.set_option("stop_after_layer", li)
    try:
        run(gnet, cfgs, x, batch, res, wave)
    finally:
        gnet.set_option("stop_after_layer", -1)
    maps = []
    for m, c in enumerate(cfgs):
        K = int(gnet.subnet_encode(c)[li][0])
        if not K:
            maps.append(None)
            continue
        dims = gnet.debug_layer_map(arr[m], batch, res, m if wave else -1, li, buf.data_ptr(), 2 * buf.numel())
        torch.cuda.synchronize()
        t = buf[:int(np.prod(dims))].reshape(dims).clone()
        assert torch.count_nonzero(t[..., K:]) == 0, (layer, m)
        maps.append(t[..., :K])
    return maps


def check(P, name, got, x, k, stride, act=None, res=None, groups=1, pool=False, what=""):
    """got, x, res: NHWC bf16.  An element may be off by its rounding to bf16 (half a step: 2^-9 of the value; twice that where the fp32
    sum lies next to a tie) and by the fp32 sum itself: every MMA step of 16 products, and the epilogue, may lose 2^-22 of the sum of
    the magnitudes."""
    for i in range(0, x.shape[0], 16):  # (double-precision maps of a few images at a time)
        xs = x[i:i + 16].permute(0, 3, 1, 2).double()
        rs = None if res is None else res[i:i + 16].permute(0, 3, 1, 2).double()
        d, K = P[name], got.shape[-1]
        R = d["w"].shape[2]
        o = (R - k) // 2
        w = d["w"][:K, :1 if groups > 1 else xs.shape[1], o:o + k, o:o + k]
        scale = (d["gamma"][:K] / torch.sqrt(d["var"][:K] + 1e-5)).view(1, -1, 1, 1)
        shift = d["beta"][:K].view(1, -1, 1, 1) - d["mean"][:K].view(1, -1, 1, 1) * scale
        y = F.conv2d(xs, w, stride=stride, padding=(k - 1) // 2, groups=groups) * scale + shift
        mag = F.conv2d(xs.abs(), w.abs(), stride=stride, padding=(k - 1) // 2, groups=groups) * scale.abs() + shift.abs()
        if rs is not None:
            y, mag = y + rs, mag + rs.abs()
        if act == "relu":
            y = torch.relu(y)
        elif act == "hswish":
            y = torch_ref.hswish(y)
        if pool:
            y, mag = F.max_pool2d(y, 3, 2, 1), F.max_pool2d(mag, 3, 2, 1)
        terms = w[0].numel()
        bound = 2.0 ** -8 * y.abs() + (terms / 16 + 8) * 2.0 ** -22 * mag
        diff = (got[i:i + 16].permute(0, 3, 1, 2).double() - y).abs()
        assert diff.shape == bound.shape, (name, what)
        worst = (diff - bound).max().item()  # (a NaN is not <= 0 either)
        assert worst <= 0, (name, what, i, worst, int((diff > bound).sum()), diff.numel())


# maps that end inside a tile, at its end and one beyond; more tiles than blocks; members of different widths; tiny: stride 1
@pytest.mark.parametrize("family,res,batch,members", [
    (wl.RESNET, 64, 1, 3), (wl.RESNET, 75, 2, 2), (wl.RESNET, 97, 1, 4), (wl.RESNET, 33, 1, 0), (wl.RESNET, 130, 1, 0), (wl.RESNET, 224, 3, 2),
    (wl.RESNET, 225, 4, 0), (wl.MBV3, 33, 2, 3), (wl.MBV3, 64, 1, 0), (wl.MBV3, 71, 2, 0), (wl.MBV3, 224, 8, 2), (wl.TINY, 32, 1, 0), (wl.TINY, 41, 2, 3),
    (wl.TINY, 8, 1, 0),
])
def test_stem_map(family, res, batch, members):
    _, _, gnet = gu.nets(family, True)
    names = [r.name for r in wl.supernet_records(family)]
    cfgs = [wl.extreme_cfg(family, True), wl.extreme_cfg(family, False)] + wl.uniform_stream(family, 4, seed=res)
    if family == wl.TINY:  # (a stem of 12 filters is a direct convolution)
        cfgs = [c for c in cfgs if int(gnet.subnet_encode(c)[0][0]) % 8 == 0]
    k, stride, act = {wl.RESNET: (7, 2, "relu"), wl.MBV3: (3, 2, "hswish"), wl.TINY: (3, 1, "relu")}[family]
    for group in ([cfgs[:members]] if members else [[c] for c in cfgs[:2]]):
        x = gu.to_device(wl.make_inputs(len(group), batch, res, seed=9, bf16=True).reshape(len(group) * batch, res, res, 3), True)
        for m, got in enumerate(maps_of(gnet, names, "stem", group, x, batch, res, members)):
            check(params(family), "stem", got, x[m * batch:(m + 1) * batch], k, stride, act, pool=family == wl.RESNET, what=(m, res))
    assert sgs.device_status() == 0


def check_resnet_blocks(gnet, cfgs, x, batch, res, wave, blocks):
    names = [r.name for r in wl.supernet_records(wl.RESNET)]
    P = params(wl.RESNET)
    get = lambda layer: maps_of(gnet, names, layer, cfgs, x, batch, res, wave)
    for s, b in blocks:
        n = f"s{s}b{b}."
        stride = 2 if s and not b else 1
        conv1, conv2, conv3 = (get(n + leaf) for leaf in ("conv1", "conv2", "conv3"))
        proj = get(n + "proj") if b == 0 else [None] * len(cfgs)
        # the block's input: the stem's pooled map, or the last block of a SubNet's stage in front of it
        fronts = ["stem"] if s == b == 0 else [f"s{s}b{b - 1}.conv3"] if b else [f"s{s - 1}b{i}.conv3" for i in range(6) if f"s{s - 1}b{i}.conv3" in names]
        inputs = [None] * len(cfgs)
        for f in fronts:
            for m, t in enumerate(get(f)):
                inputs[m] = t if t is not None else inputs[m]
        for m in range(len(cfgs)):
            if conv1[m] is None:
                continue
            what = (m, res, batch, wave)
            check(P, n + "conv1", conv1[m], inputs[m], 1, 1, "relu", what=what)
            check(P, n + "conv2", conv2[m], conv1[m], 3, stride, "relu", what=what)
            if b == 0:
                check(P, n + "proj", proj[m], inputs[m], 1, stride, what=what)
            check(P, n + "conv3", conv3[m], conv2[m], 1, 1, "relu", res=proj[m] if b == 0 else inputs[m], what=what)


# maps of 16, 8, 4, 2 (swapped tiles), 18, 9, 5, 3, 56 .. 7 (two members in a tile), 49 x 49 .. 7; several images a member
@pytest.mark.parametrize("res,batch,members", [(64, 1, 5), (72, 1, 6), (224, 1, 7), (193, 1, 3), (72, 3, 3), (224, 16, 2)])
def test_grouped_layers_of_a_wave(res, batch, members):
    _, _, gnet = gu.nets(wl.RESNET, True)
    cfgs = [wl.extreme_cfg(wl.RESNET, True), wl.extreme_cfg(wl.RESNET, False)] + wl.uniform_stream(wl.RESNET, members - 2, seed=res)
    x = gu.to_device(wl.make_inputs(members, batch, res, seed=5, bf16=True).reshape(members * batch, res, res, 3), True)
    check_resnet_blocks(gnet, cfgs, x, batch, res, 1, [(0, 0), (0, 1), (1, 0), (2, 3), (3, 0), (3, 1)])
    assert sgs.device_status() == 0


# one image: latency kernel, split reductions, projection and first convolution in one launch; 16: the first stage on the grouped kernel
@pytest.mark.parametrize("res,batch,grouped", [(64, 1, False), (224, 1, False), (97, 3, False), (224, 16, True)])
def test_layers_of_a_single_query(res, batch, grouped):
    _, _, gnet = gu.nets(wl.RESNET, True)
    cfg = wl.extreme_cfg(wl.RESNET, True)
    x = gu.to_device(wl.make_inputs(1, batch, res, seed=5, bf16=True).reshape(batch, res, res, 3), True)
    gnet.set_option("drop_plans", 1)
    check_resnet_blocks(gnet, [cfg], x, batch, res, 0, [(0, 0), (0, 1), (1, 0), (3, 1)])
    assert (gnet.get_counter("grouped_convs") > 0) == grouped
    assert sgs.device_status() == 0


def test_more_tiles_for_a_block_than_it_keeps_records_of():
    # 776 images of 56x56 pixels: 19 012 tiles for 148 blocks, 128.5 each; the records of the last ones are worked out on the way
    _, _, gnet = gu.nets(wl.RESNET, True)
    cfg, batch, res = wl.extreme_cfg(wl.RESNET, True), 776, 224
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(batch, res, res, 3, device="cuda", generator=g).to(torch.bfloat16)
    net = sgs.SuperNet(wl.RESNET, gu.nets(wl.RESNET, True)[0], sgs.SGS_BF16)  # (its workspaces, 5 GB, go with it)
    try:
        names = [r.name for r in wl.supernet_records(wl.RESNET)]
        maps = {n: maps_of(net, names, n, [cfg], x, batch, res, 0)[0] for n in ("stem", "s0b0.proj", "s0b0.conv1", "s0b0.conv2", "s0b0.conv3")}
        assert net.get_counter("grouped_convs") > 0
        P = params(wl.RESNET)
        check(P, "stem", maps["stem"], x, 7, 2, "relu", pool=True)
        check(P, "s0b0.proj", maps["s0b0.proj"], maps["stem"], 1, 1)
        check(P, "s0b0.conv1", maps["s0b0.conv1"], maps["stem"], 1, 1, "relu")
        check(P, "s0b0.conv2", maps["s0b0.conv2"], maps["s0b0.conv1"], 3, 1, "relu")
        check(P, "s0b0.conv3", maps["s0b0.conv3"], maps["s0b0.conv2"], 1, 1, "relu", res=maps["s0b0.proj"])
    finally:
        net.close()
    assert sgs.device_status() == 0


@pytest.mark.parametrize("res,members", [(64, 4), (71, 3), (224, 3)])
def test_mobilenet_layers_of_a_wave(res, members):
    # stages without squeeze-excite (it scales the depthwise map in place); all three depthwise kernel sizes
    _, _, gnet = gu.nets(wl.MBV3, True)
    names = [r.name for r in wl.supernet_records(wl.MBV3)]
    P = params(wl.MBV3)
    cfgs = [wl.extreme_cfg(wl.MBV3, True), wl.extreme_cfg(wl.MBV3, False)] + wl.uniform_stream(wl.MBV3, members - 2, seed=res)
    x = gu.to_device(wl.make_inputs(members, 1, res, seed=5, bf16=True).reshape(members, res, res, 3), True)
    for s, b, front, stride, act in ((0, 0, "first.pw", 2, "relu"), (0, 1, "s0b0.project", 1, "relu"), (2, 1, "s2b0.project", 1, "hswish")):
        n = f"s{s}b{b}."
        front, expand, dw, project = (maps_of(gnet, names, layer, cfgs, x, 1, res, 1) for layer in (front, n + "expand", n + "dw", n + "project"))
        for m, c in enumerate(cfgs):
            k = int(c.kernel[s][b])
            check(P, n + "expand", expand[m], front[m], 1, 1, act, what=m)
            check(P, n + "dw", dw[m], expand[m], k, stride, act, groups=expand[m].shape[-1], what=m)
            check(P, n + "project", project[m], dw[m], 1, 1, None, res=front[m] if stride == 1 else None, what=m)
    assert sgs.device_status() == 0


def test_layer_maps_refuse_what_was_not_run():
    _, _, gnet = gu.nets(wl.RESNET, True)
    arr = wl.cfg_array([wl.extreme_cfg(wl.RESNET, False)])
    buf = torch.zeros(64, dtype=torch.bfloat16, device="cuda")
    for member, layer, size in ((5000, 1, 128), (-1, 10000, 128), (-2, 1, 128), (-1, 1, 2)):
        with pytest.raises(sgs.SgsError):
            gnet.debug_layer_map(arr[0], 1, 80, member, layer, buf.data_ptr(), size)
    for bad in (-2, 10000, gnet.n_layers - 1):  # (the last stored layer is the classifier)
        with pytest.raises(sgs.SgsError):
            gnet.set_option("stop_after_layer", bad)


def test_the_comparison_sees_one_wrong_tap_and_one_wrong_pixel():
    # mistakes planted in the reference: a tap of one filter left out, one pixel of the image's border changed
    _, _, gnet = gu.nets(wl.RESNET, True)
    names = [r.name for r in wl.supernet_records(wl.RESNET)]
    cfgs, res = [wl.extreme_cfg(wl.RESNET, True), wl.extreme_cfg(wl.RESNET, False)], 64
    x = gu.to_device(wl.make_inputs(2, 1, res, seed=5, bf16=True).reshape(2, res, res, 3), True)
    stem = maps_of(gnet, names, "stem", cfgs, x, 1, res, 1)
    conv1 = maps_of(gnet, names, "s0b0.conv1", cfgs, x, 1, res, 1)
    P = params(wl.RESNET)
    for name, got, source, k, stride, pool in (("stem", stem[1], x[1:], 7, 2, True), ("s0b0.conv1", conv1[0], stem[0], 1, 1, False)):
        check(P, name, got, source, k, stride, "relu", pool=pool)
        wrong = dict(P[name], w=P[name]["w"].clone())
        wrong["w"][3, 1, -1, -1] = 0
        with pytest.raises(AssertionError):
            check({name: wrong}, name, got, source, k, stride, "relu", pool=pool)
        changed = source.clone()
        changed[0, -1, -1] += 1
        with pytest.raises(AssertionError):
            check(P, name, got, changed, k, stride, "relu", pool=pool)
