"""The device side of clustering and transfer at its edges, against the
oracle: row lengths around the 32-cell scans, buffers wider than a box side,
new hierarchies shallower, as deep as and deeper than the old one (finest
cells found through the covered list, or through the box of a single level),
several vectors, repeated calls with growing scratch.  Boxes are integers and
must be equal; the transfer's bound is that of the other transfer tests,
1e-14 of max |u| (two FP64 operations per axis)."""
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import regrid as R  # noqa: E402
from paper_1302_6303_gb300 import workloads as W  # noqa: E402
from regrid_cases import random_hierarchy  # noqa: E402


@pytest.fixture(scope="module")
def nrd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1302_6303_gb300 import nrd as m
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def ctx_for(nrd, h):
    ctx = nrd.Context(nmg=1)
    ctx.set_hierarchy_from(h)
    ctx.set_material(dev(np.ones(h.ncells, np.float32)))
    return ctx


def as_lists(levels):
    return [[(tuple(lo), tuple(hi)) for lo, hi in lev] for lev in levels]


@pytest.mark.parametrize("n0", [(33, 5, 4), (31, 7, 3), (32, 4, 6), (1, 9, 8), (65, 3, 3)])
@pytest.mark.parametrize("levels", [1, 2])
def test_boxes(nrd, n0, levels):
    rng = np.random.default_rng(sum(n0) + levels)
    h = W.uniform(n0) if levels == 1 else random_hierarchy(rng, n0, 2, count=2, side_lo=2,
                                                           side_hi=4)
    tags = (rng.random(h.ncells) < 0.08).astype(np.uint8) * 2
    ctx = ctx_for(nrd, h)
    for buf, eff, mn, mx, ml in [(0, 0.6, 2, 8, 2), (1, 0.7, 2, 32, 3), (6, 0.7, 4, 16, 3)]:
        got = ctx.regrid_boxes(dev(tags), 2, buf, eff, mn, mx, ml)
        exp = R.regrid_boxes(h, tags, tag_bits=2, buffer=buf, efficiency=eff, min_side=mn,
                             max_side=mx, max_levels=ml)
        assert as_lists(got) == as_lists(exp)


@pytest.mark.parametrize("old", [1, 2, 3])
@pytest.mark.parametrize("new", [1, 2, 3])
def test_transfer_depths(nrd, old, new):
    rng = np.random.default_rng(10 * old + new)
    n0 = (9, 6, 7)
    mk = lambda L: W.uniform(n0) if L == 1 else random_hierarchy(rng, n0, L)  # noqa: E731
    a, b = mk(old), mk(new)
    ca, cb = ctx_for(nrd, a), ctx_for(nrd, b)
    for nvec in (1, 3):
        u = rng.uniform(0.1, 2.0, (nvec, 2 * a.ncells))
        out = ca.transfer_to(cb, dev(u)).cpu().numpy()
        for v, o in zip(u, out):
            exp = R.transfer(a, b, v)
            assert np.abs(o - exp).max() <= 1e-14 * np.abs(exp).max()


def test_transfer_threads(nrd):
    """Two threads, each with a stream and a destination of its own, transfer
    from one context whose scratch they share; the values are those of the
    same calls one after the other."""
    rng = np.random.default_rng(5)
    n0 = (17, 12, 9)
    a, b = random_hierarchy(rng, n0, 2), random_hierarchy(rng, n0, 3)
    ca = ctx_for(nrd, a)
    cb = [ctx_for(nrd, b), ctx_for(nrd, b)]
    us = [[dev(rng.uniform(0.1, 2.0, (nv, 2 * a.ncells))) for nv in (1, 4, 2, 6)] for _ in cb]
    exp = [[ca.transfer_to(c, u) for u in w] for c, w in zip(cb, us)]
    torch.cuda.synchronize()
    got = [[], []]

    def work(t):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(5):
                got[t] = [ca.transfer_to(cb[t], u) for u in us[t]]

    th = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    torch.cuda.synchronize()
    for g, e in zip(got, exp):
        assert len(g) == len(e) and all(torch.equal(x, y) for x, y in zip(g, e))


@pytest.mark.parametrize("cluster", ["tag side", "tag default", "copy side"])
def test_tags_from_another_stream(nrd, cluster):
    """Tags written late on a side stream, by nrd_tag or by torch, are the ones
    clustered, from that stream or (nrd_tag's) from the default one: the boxes
    are those of the same tags made and clustered on the default stream."""
    h = W.uniform(24)
    u = dev(W.front_state(h, seed=4, noise=0.0, front=0.4, width=0.1))
    ctx = ctx_for(nrd, h)
    ref = ctx.tag(u, thr_r=0.1)
    boxes = lambda t: as_lists(ctx.regrid_boxes(t, 4, 1, 0.7, 4, 16, 2))  # noqa: E731
    exp = boxes(ref)
    assert len(exp) == 2
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for _ in range(2):   # (untagged bytes are what an early read would find)
            torch.zeros(h.ncells, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        if cluster == "copy side":
            tags = torch.zeros_like(ref)
            torch.cuda._sleep(200_000_000)
            tags.copy_(ref)
        else:
            torch.cuda._sleep(200_000_000)
            tags = ctx.tag(u, thr_r=0.1)
        if cluster != "tag default":
            got = boxes(tags)
    if cluster == "tag default":
        got = boxes(tags)
    assert got == exp


def test_transfer_does_not_wait_for_another(nrd):
    """A transfer returns while another thread's, from the same context, still
    waits for earlier work on its own stream."""
    rng = np.random.default_rng(6)
    n0 = (17, 12, 9)
    a, b = random_hierarchy(rng, n0, 2), random_hierarchy(rng, n0, 3)
    ca, cb = ctx_for(nrd, a), [ctx_for(nrd, b), ctx_for(nrd, b)]
    u = dev(rng.uniform(0.1, 2.0, 2 * a.ncells))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    exp = []
    for s, c in zip(streams, cb):   # kernels loaded, output memory in each stream's pool
        with torch.cuda.stream(s):
            exp.append(ca.transfer_to(c, u).cpu())
    torch.cuda.synchronize()
    begun, ended, got = threading.Event(), threading.Event(), [None, None]

    def late():
        with torch.cuda.stream(streams[0]):
            torch.cuda._sleep(4_000_000_000)   # about two seconds
            begun.set()
            got[0] = ca.transfer_to(cb[0], u)
        ended.set()

    th = threading.Thread(target=late)
    th.start()
    begun.wait()
    time.sleep(0.3)
    with torch.cuda.stream(streams[1]):
        got[1] = ca.transfer_to(cb[1], u)
    first = not ended.is_set()
    th.join()
    torch.cuda.synchronize()
    assert first
    assert all(torch.equal(g.cpu(), e) for g, e in zip(got, exp))


@pytest.mark.parametrize("n0,levels", [
    ((16, 32, 16), 1), ((17, 32, 16), 1), ((33, 17, 15), 1), ((8193, 1, 1), 1), ((1, 97, 89), 1),
    ((3, 4, 700), 1), ((40, 9, 25), 1), ((17, 18, 17), 1), ((9, 10, 700), 1), ((16, 32, 16), 2), ((17, 32, 16), 2), ((40, 9, 25), 2)])
def test_boxes_both_forms(nrd, n0, levels):
    """Index spaces on both sides of the line between the host and the device
    form of the fields (about 20^3 cells, fewer with a wider buffer, more for a
    long box), level 0 on one and level 1 on the other among them, against the
    oracle."""
    rng = np.random.default_rng(sum(n0) + levels)
    h = W.uniform(n0) if levels == 1 else random_hierarchy(rng, n0, 2, count=2, side_lo=2,
                                                           side_hi=4)
    tags = (rng.random(h.ncells) < 0.01).astype(np.uint8) * 2
    ctx = ctx_for(nrd, h)
    for buf, eff, mn, mx, ml in [(0, 0.6, 2, 16, 2), (1, 0.7, 4, 32, 2 + (levels == 2)),
                                 (5, 0.7, 4, 16, 2)]:
        got = ctx.regrid_boxes(dev(tags), 2, buf, eff, mn, mx, ml)
        exp = R.regrid_boxes(h, tags, tag_bits=2, buffer=buf, efficiency=eff, min_side=mn,
                             max_side=mx, max_levels=ml)
        assert as_lists(got) == as_lists(exp)


def test_tags_of_a_captured_call(nrd):
    """nrd_tag in a CUDA graph, replayed on new states: the clustering takes the
    replay's tags."""
    h = W.uniform(24)
    u = dev(W.front_state(h, seed=4, noise=0.0, front=0.4, width=0.1))
    late = dev(W.front_state(h, seed=4, noise=0.0, front=0.6, width=0.1))
    ctx = ctx_for(nrd, h)
    boxes = lambda t: as_lists(ctx.regrid_boxes(t, 4, 1, 0.7, 4, 16, 2))  # noqa: E731
    exp = [boxes(ctx.tag(x, thr_r=0.1)) for x in (u, late)]
    assert exp[0] != exp[1]
    v, s, g = u.clone(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        tags = ctx.tag(v, thr_r=0.1)
    with torch.cuda.stream(s):
        for x, e in zip((u, late), exp):
            torch.cuda._sleep(100_000_000)
            v.copy_(x)
            g.replay()
            assert boxes(tags) == e
