"""Device buffers kept from a released handle for the next one on its stream:
results stay right when handles are packed, used and released without waiting,
on one stream, on two, under graph replay and from several threads, and what is
kept stays bounded and goes back on request."""
import threading

import numpy as np
import pytest

from paper_2609_33977_gb300 import workload as wl
from tests._gpu_util import to_bits, to_dev

pytestmark = pytest.mark.gpu
OUT, INP, T = 1536, 2048, 24


@pytest.fixture(scope="module")
def gs(built_lib):
    import torch
    assert torch.cuda.is_available(), "the -m gpu tests need a CUDA device"
    from paper_2609_33977_gb300 import groupsparse
    return groupsparse


@pytest.fixture(scope="module")
def data(gs):
    """(W, x, masks, the bits of y for each mask), each y from a handle that lives through its call."""
    import torch
    W = to_dev(wl.random_weight_bits(OUT, INP, seed=1))
    x = to_dev(wl.random_activation_bits(T, INP, seed=2))
    masks = [torch.from_numpy(wl.random_mask(OUT, INP // 256, 0.5, seed=10 + i)).cuda() for i in range(6)]
    ref, handles = [], []
    for m in masks:
        handles.append(gs.pack(W, m))
        ref.append(to_bits(gs.linear(x, handles[-1])))
    torch.cuda.synchronize()
    return W, x, masks, ref


def cycle(gs, data, n, before_linear=None):
    W, x, masks, _ = data
    ys = []
    for i in range(n):
        p = gs.pack(W, masks[i % len(masks)])
        if before_linear:
            before_linear()
        ys.append((gs.linear(x, p, algo=gs.ALGO_DECODE if i % 2 else gs.ALGO_AUTO), gs.unpack(p)))
        p.free()
    return ys


def check(gs, data, ys, ref_by_algo):
    for i, (y, _) in enumerate(ys):
        k = i % len(data[2])
        assert np.array_equal(to_bits(y), ref_by_algo[i % 2][k]), i


@pytest.fixture(scope="module")
def refs(gs, data):
    W, x, masks, ref = data
    handles = [gs.pack(W, m) for m in masks]
    return ref, [to_bits(gs.linear(x, p, algo=gs.ALGO_DECODE)) for p in handles]


def test_repacking_on_one_stream_reuses_buffers_and_keeps_results(gs, data, refs):
    import torch
    cycle(gs, data, 6)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    # a kernel in front of each call keeps the previous handle's work in flight while the next is packed
    ys = cycle(gs, data, 18, before_linear=lambda: torch.cuda._sleep(200_000))
    torch.cuda.synchronize()
    check(gs, data, ys, refs)
    assert torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved() == held   # no new device memory


def test_handle_used_on_a_second_stream_is_not_reused_early(gs, data, refs):
    import torch
    W, x, masks, _ = data
    other = torch.cuda.Stream()
    ys = []
    for i in range(6):
        p = gs.pack(W, masks[i])
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            torch.cuda._sleep(2_000_000)
            ys.append(gs.linear(x, p))
        p.free()                        # work on `other` still queued
        q = gs.pack(W, masks[(i + 1) % 6])   # would take the buffers, were they kept
        q.free()
    torch.cuda.synchronize()
    for i, y in enumerate(ys):
        assert np.array_equal(to_bits(y), refs[0][i]), i


def test_handle_captured_into_a_graph_is_not_reused_early(gs, data, refs):
    import torch
    W, x, masks, _ = data
    y = torch.empty((T, OUT), dtype=torch.bfloat16, device="cuda")
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        p = gs.pack(W, masks[0])
        gs.linear_into(x, p, y)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            torch.cuda._sleep(2_000_000)
            gs.linear_into(x, p, y)
    y.zero_()
    torch.cuda.synchronize()
    g.replay()                          # on the default stream
    p.free()
    with torch.cuda.stream(stream):
        q = gs.pack(W, masks[1])
    torch.cuda.synchronize()
    assert np.array_equal(to_bits(y), refs[0][0])
    q.free()


def test_threads_with_streams_of_their_own_and_a_shared_one(gs, data, refs):
    import torch
    shared = torch.cuda.Stream()
    out, errors = {}, []

    def work(k):
        try:
            s = shared if k < 2 else torch.cuda.Stream()
            with torch.cuda.stream(s):
                out[k] = cycle(gs, data, 12)
            s.synchronize()
        except Exception as e:   # reported below
            errors.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert not errors, errors
    torch.cuda.synchronize()
    for k in range(4):
        check(gs, data, out[k], refs)


def test_what_is_kept_is_bounded(gs):
    import torch
    free_b, total = torch.cuda.mem_get_info()
    W = torch.zeros((16384, 16384), dtype=torch.bfloat16, device="cuda")   # 512 MB packed when all groups are kept
    mask = torch.ones((16384, 64), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    handles = [gs.pack(W, mask) for _ in range(6)]
    for p in handles:
        p.free()
    torch.cuda.synchronize()
    assert free0 - torch.cuda.mem_get_info()[0] <= total // 128 + (64 << 20)
    gs.trim()
    assert torch.cuda.mem_get_info()[0] >= free0
