"""GPU parity of persistent execution (the whole stream as one launch of the SubNet kernel) against the CPU oracle.

Same tolerance as the other bf16 parity tests: max|err| <= 2e-2 * max|ref| per output row, against the oracle run
with the same storage rounding points and against the plain fp32 oracle.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

TOL_BF16 = 2e-2


def _run(gnet, cfgs, d_in, res, host=False, cache=1, window_q=4):
    n = len(cfgs)
    stream = torch.cuda.Stream()
    opts = sgs.StreamOpts(cache_enabled=cache, window_q=window_q, cache_budget_bytes=0, use_graphs=0, record_latency=0,
                          concurrency=1, wave=0, policy=0, persistent=1)
    if host:
        h_out = np.zeros((n, 1000), dtype=np.float32)
        h_in = d_in.cpu().view(torch.int16).numpy()
        st = gnet.stream_run(cfgs, h_in, 1, res, h_out, opts, stream.cuda_stream, host=True)
        return h_out, st
    d_out = torch.zeros((n, 1000), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    st = gnet.stream_run(cfgs, d_in.data_ptr(), 1, res, d_out.data_ptr(), opts, stream.cuda_stream)
    return d_out.cpu().numpy(), st


@pytest.mark.parametrize("res,n", [(64, 9), (96, 7)])
def test_persistent_stream_matches_checker(res, n):
    # uniform configs plus the smallest and the largest SubNet; fewer queries than SMs, so every block serves at most one
    _, onet, gnet = gu.nets(wl.MBV3, True)
    cfgs = wl.uniform_stream(wl.MBV3, n - 2, seed=21) + [wl.extreme_cfg(wl.MBV3, False), wl.extreme_cfg(wl.MBV3, True)]
    xs = wl.make_inputs(n, 1, res, seed=6, bf16=True)
    d_in = gu.to_device(xs.reshape(n, res, res, 3), True)
    got, st = _run(gnet, cfgs, d_in, res)
    assert st.kernel_launches == 1 and st.n_queries == n
    assert np.all(np.isfinite(got))
    for t in range(n):
        ref = onet.forward(cfgs[t], xs[t], oracle.BF16_STORE)
        assert gu.rel_err(got[t:t + 1], ref) <= TOL_BF16, t
        plain = onet.forward(cfgs[t], xs[t], oracle.FP32)
        assert gu.rel_err(got[t:t + 1], plain) <= TOL_BF16, t
    again, _ = _run(gnet, cfgs, d_in, res)
    np.testing.assert_array_equal(again, got)          # which block serves a query does not change its bits
    hosted, _ = _run(gnet, cfgs, d_in, res, host=True)
    np.testing.assert_array_equal(hosted, got)


def test_persistent_stream_many_queries_per_block_equals_the_wave_path():
    # 400 queries on 148 blocks: every block serves several queries out of the same scratch area.  The layer-by-layer
    # wave path (itself checked against the oracle elsewhere) computes the same layers with other kernels: the two
    # agree within the parity bound on every query, and sampled queries are compared with the oracle directly.
    _, onet, gnet = gu.nets(wl.MBV3, True)
    n, res = 400, 64
    cfgs = wl.uniform_stream(wl.MBV3, n, seed=33)
    xs = wl.make_inputs(n, 1, res, seed=8, bf16=True)
    d_in = gu.to_device(xs.reshape(n, res, res, 3), True)
    got, st = _run(gnet, cfgs, d_in, res)
    assert st.kernel_launches == 1
    stream = torch.cuda.Stream()
    d_out = torch.zeros((n, 1000), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    wopts = sgs.StreamOpts(cache_enabled=1, window_q=4, cache_budget_bytes=0, use_graphs=0, record_latency=0,
                           concurrency=2, wave=32)
    wst = gnet.stream_run(cfgs, d_in.data_ptr(), 1, res, d_out.data_ptr(), wopts, stream.cuda_stream)
    waves = d_out.cpu().numpy()
    for t in range(n):
        assert gu.rel_err(got[t:t + 1], waves[t:t + 1]) <= TOL_BF16, t
    for t in (0, 147, 148, 313, 399):
        ref = onet.forward(cfgs[t], xs[t], oracle.BF16_STORE)
        assert gu.rel_err(got[t:t + 1], ref) <= TOL_BF16, t
    assert st.useful_flops == wst.useful_flops and st.weight_bytes == wst.weight_bytes


def test_weight_buffer_in_shared_memory_changes_no_bit():
    # With the cache on, every block keeps the chosen SubGraph's first pointwise layers in shared memory and multiplies
    # them in place; filters and channels of a query beyond the box still come through the ring.  The arithmetic of an
    # output column does not depend on where its filter came from, so logits are bit-identical with the buffer off,
    # small (a box that ends inside a layer's neighbours) and at its largest; the accounting is against what is held.
    _, _, gnet = gu.nets(wl.MBV3, True)
    n, res = 200, 96
    cfgs = wl.markov_stream(n, seed=12, family=wl.MBV3)
    d_in = gu.to_device(wl.make_inputs(n, 1, res, seed=13, bf16=True).reshape(n, res, res, 3), True)
    off, st_off = _run(gnet, cfgs, d_in, res, cache=0)
    assert st_off.hit_ratio == 0 and st_off.hbm_weight_bytes == st_off.weight_bytes
    try:
        for kb in (8, 40, 56):
            gnet.set_option("persistent_held_kb", kb)
            for q in (1, 4):
                on, st_on = _run(gnet, cfgs, d_in, res, cache=1, window_q=q)
                np.testing.assert_array_equal(on, off)
                assert 0 < st_on.hit_ratio < 1 and st_on.hbm_weight_bytes < st_on.weight_bytes
                assert st_on.cache_updates == 1
        gnet.set_option("persistent_held_kb", 0)
        none, st_none = _run(gnet, cfgs, d_in, res, cache=1)
        np.testing.assert_array_equal(none, off)
        assert st_none.hbm_weight_bytes == st_none.weight_bytes
        with pytest.raises(sgs.SgsError):
            gnet.set_option("persistent_held_kb", 4096)
    finally:
        gnet.set_option("persistent_held_kb", 16)


@pytest.mark.parametrize("team", [1, 2, 4, 8, 16])
def test_weight_buffer_is_used_by_every_team(team):
    # Layers whose filters are split over a team's blocks (maps of 64x64 images have 8 pixel tiles at most) multiply the part of the
    # box that a tile covers: the same bits as without a buffer, and the same figures for every team.
    _, _, gnet = gu.nets(wl.MBV3, True)
    n, res = 20, 64
    cfgs = wl.markov_stream(n - 2, seed=12, family=wl.MBV3) + [wl.extreme_cfg(wl.MBV3, False), wl.extreme_cfg(wl.MBV3, True)]
    d_in = gu.to_device(wl.make_inputs(n, 1, res, seed=13, bf16=True).reshape(n, res, res, 3), True)
    try:
        gnet.set_option("persistent_team", 1)
        off, _ = _run(gnet, cfgs, d_in, res, cache=0)
        for kb in (16, 56):
            gnet.set_option("persistent_held_kb", kb)
            gnet.set_option("persistent_team", 1)
            _, st_one = _run(gnet, cfgs, d_in, res)
            gnet.set_option("persistent_team", team)
            on, st_on = _run(gnet, cfgs, d_in, res)
            np.testing.assert_array_equal(on, off)
            assert 0 < st_on.hbm_weight_bytes < st_on.weight_bytes
            assert (st_on.hit_ratio, st_on.hbm_weight_bytes) == (st_one.hit_ratio, st_one.hbm_weight_bytes)
    finally:
        gnet.set_option("persistent_held_kb", 16)
        gnet.set_option("persistent_team", 0)


def test_persistent_stream_full_resolution_sampled():
    _, onet, gnet = gu.nets(wl.MBV3, True)
    n, res = 160, 224
    cfgs = wl.uniform_stream(wl.MBV3, n, seed=3)
    xs = wl.make_inputs(n, 1, res, seed=4, bf16=True)
    d_in = gu.to_device(xs.reshape(n, res, res, 3), True)
    got, _ = _run(gnet, cfgs, d_in, res)
    assert np.all(np.isfinite(got))
    for t in (0, 150, 159):
        ref = onet.forward(cfgs[t], xs[t], oracle.BF16_STORE)
        assert gu.rel_err(got[t:t + 1], ref) <= TOL_BF16, t


def test_persistent_refusals():
    _, _, rnet = gu.nets(wl.RESNET, True)
    cfgs = wl.uniform_stream(wl.RESNET, 2, seed=1)
    d_in = gu.to_device(wl.make_inputs(2, 1, 64, seed=1, bf16=True).reshape(2, 64, 64, 3), True)
    with pytest.raises(sgs.SgsError) as e:
        _run(rnet, cfgs, d_in, 64)
    assert e.value.status == sgs.binding.SGS_EUNSUPPORTED
    _, _, gnet = gu.nets(wl.MBV3, True)
    mcfgs = wl.uniform_stream(wl.MBV3, 2, seed=1)
    d_out = torch.zeros((4, 1000), dtype=torch.float32, device="cuda")
    d_in2 = gu.to_device(wl.make_inputs(2, 2, 64, seed=1, bf16=True).reshape(4, 64, 64, 3), True)
    opts = sgs.StreamOpts(cache_enabled=0, window_q=1, persistent=1)
    with pytest.raises(sgs.SgsError) as e:
        gnet.stream_run(mcfgs, d_in2.data_ptr(), 2, 64, d_out.data_ptr(), opts, 0)
    assert e.value.status == sgs.binding.SGS_EINVAL
    # an empty stream is fine
    st = gnet.stream_run(mcfgs[:0], d_in2.data_ptr(), 1, 64, d_out.data_ptr(), opts, 0)
    assert st.n_queries == 0


@pytest.mark.parametrize("team,res,n", [(2, 64, 3), (4, 96, 4), (8, 72, 3), (16, 64, 2), (16, 40, 9), (2, 104, 80)])
def test_teams_of_blocks_agree_with_single_blocks(team, res, n):
    # layers with fewer tiles, rows, pixels or outputs than the team has threads or blocks (a 2x2 map, one pixel tile); more
    # queries than teams; the smallest and the largest SubNet.  A query's bits do not depend on the team.
    _, onet, gnet = gu.nets(wl.MBV3, True)
    cfgs = wl.uniform_stream(wl.MBV3, n - 2, seed=5) + [wl.extreme_cfg(wl.MBV3, False), wl.extreme_cfg(wl.MBV3, True)]
    xs = wl.make_inputs(n, 1, res, seed=6, bf16=True)
    d_in = gu.to_device(xs.reshape(n, res, res, 3), True)
    try:
        gnet.set_option("persistent_team", 1)
        alone, _ = _run(gnet, cfgs, d_in, res)
        gnet.set_option("persistent_team", team)
        got, st = _run(gnet, cfgs, d_in, res)
        again, _ = _run(gnet, cfgs, d_in, res)
        with pytest.raises(sgs.SgsError):
            gnet.set_option("persistent_team", 3)
    finally:
        gnet.set_option("persistent_team", 0)
    assert st.kernel_launches == 1
    np.testing.assert_array_equal(again, got)
    np.testing.assert_array_equal(got, alone)
    for t in (0, n - 2, n - 1):
        assert gu.rel_err(got[t:t + 1], onet.forward(cfgs[t], xs[t], oracle.BF16_STORE)) <= TOL_BF16, t
    assert sgs.device_status() == 0


@pytest.mark.parametrize("res", [224, 72])
def test_logits_do_not_depend_on_the_number_of_queries(res):
    # a query alone, in calls of more and more queries (teams of 16 blocks down to one) and with every team asked for: the same
    # bits.  224: pooled maps of 28, 14 and 7 pixels a side; 72: 9, 5 and 3, fewer pixels than shares.
    _, _, gnet = gu.nets(wl.MBV3, True)
    n = 170
    cfgs = [wl.extreme_cfg(wl.MBV3, False), wl.extreme_cfg(wl.MBV3, True)] + wl.uniform_stream(wl.MBV3, n - 2, seed=12)
    d_in = gu.to_device(wl.make_inputs(n, 1, res, seed=3, bf16=True).reshape(n, res, res, 3), True)
    gnet.set_option("persistent_team", 1)
    try:
        ref, _ = _run(gnet, cfgs, d_in, res, cache=0)
        for team in (2, 4, 8, 16):
            gnet.set_option("persistent_team", team)
            got, _ = _run(gnet, cfgs[:40], d_in, res, cache=0)
            np.testing.assert_array_equal(got, ref[:40])
    finally:
        gnet.set_option("persistent_team", 0)
    for m in (1, 2, 9, 33, 70, 140, 170):
        got, _ = _run(gnet, cfgs[:m], d_in, res, cache=0)
        np.testing.assert_array_equal(got, ref[:m])


@pytest.mark.parametrize("res,n", [(64, 149), (64, 170), (96, 149), (128, 75)])
def test_the_chosen_team_is_not_slower_than_the_best_one(res, n):
    # small images, a few more queries than there are teams: a second round of large teams takes as long as the first.  Device times,
    # the best of five; the rule's worst case over a grid of calls is 1.24; with constants fitted at 224x224 these took up to 1.52.
    _, _, gnet = gu.nets(wl.MBV3, True)
    cfgs = wl.uniform_stream(wl.MBV3, n, seed=11)
    d_in = gu.to_device(wl.make_inputs(n, 1, res, seed=3, bf16=True).reshape(n, res, res, 3), True)
    times = {}
    try:
        for team in (1, 2, 4, 0):
            gnet.set_option("persistent_team", team)
            times[team] = min(_run(gnet, cfgs, d_in, res)[1].total_ms for _ in range(5))
    finally:
        gnet.set_option("persistent_team", 0)
    assert times[0] <= 1.24 * min(times.values()), times
