"""Arrays that other streams still read when a handle is freed are given back
after those reads: Huffman-shaped trees, which live on a stream of the
library's, under queries queued on the caller's streams, and the parts of a
merge on another stream than theirs."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import from_dev_u64, to_dev

pytestmark = pytest.mark.gpu

SPIN = 100_000_000  # clock cycles, about 50 ms


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("sigma", [300, 1 << 16])
@pytest.mark.parametrize("how", ["access", "rank", "select", "multi"])
def test_huffman_tree_freed_behind_queued_queries(wt, sigma, how):
    import torch
    n, q = 200_003, 4096
    S = synth.zipf(5, n, sigma, 1.1, 4)
    rng = np.random.default_rng(6)
    x = rng.integers(0, n, q).astype(np.uint64)
    c = S[x].astype(np.uint32)
    one = np.ones(q, np.uint64)
    exp = {"access": c.astype(np.uint64), "rank": oracle.rank(S, sigma, c, x),
           "select": oracle.select(S, sigma, c, one),
           "multi": oracle.rank(S, sigma, c, x)}[how]
    side, build = torch.cuda.Stream(), torch.cuda.Stream()
    h = wt.huff_wt_build(to_dev(S), sigma)
    h.sync()
    dx, dc, dk = to_dev(x), to_dev(c), to_dev(one)
    out = torch.zeros(q, dtype=torch.int64, device="cuda")
    multi = (torch.zeros(q, dtype=torch.int32, device="cuda"),
             torch.ones(q, dtype=torch.uint8, device="cuda"), dc, dx, out)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(SPIN)
        if how == "access":
            h.access(dx, out)
        elif how == "rank":
            h.rank(dc, dx, out)
        elif how == "select":
            h.select(dc, dk, out)
        else:
            wt.query_multi([h], *multi)
    h.free()
    assert side.query()  # the queries, queued behind the spin, are over
    # memory given back is taken by the next build on another stream
    with torch.cuda.stream(build):
        T = synth.zipf(7, n, sigma, 1.1, 4)
        h2 = wt.huff_wt_build(to_dev(T), sigma)
        h2.sync()
    assert np.array_equal(from_dev_u64(out), exp)
    h2.free()


def test_parts_freed_behind_a_queued_merge(wt):
    import torch
    n, sigma = 1 << 24, 256
    S = synth.zipf(9, n, sigma, 1.1, 1)
    ob, oz = oracle.wm_build(S, sigma)
    build, merge = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(build):
        parts = [wt.wm_build(to_dev(S[a:b].copy()), sigma) for a, b in ((0, n // 3), (n // 3, n))]
        build.synchronize()
    with torch.cuda.stream(merge):
        h = wt.dd_merge(parts)
    parts[0].free()  # waits for its stream, which waits for the merge
    assert merge.query()
    parts[1].free()
    with torch.cuda.stream(build):
        again = wt.wm_build(to_dev(S[::-1].copy()), sigma)
        again.sync()
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
    h.free()
    again.free()


def test_queries_of_several_streams(wt):
    """Every stream's queries are waited for, by the release only: a stream's
    last ones after earlier ones on it and on others, and trees that share a
    launch."""
    import torch
    n, sigma, q = 150_001, 500, 1000
    S = synth.zipf(15, n, sigma, 1.1, 2)
    x = np.random.default_rng(16).integers(0, n, q).astype(np.uint64)
    dx = to_dev(x)
    hs = [wt.huff_wt_build(to_dev(S), sigma) for _ in range(2)]
    for h in hs:
        h.sync()
    zero = torch.zeros(q, dtype=torch.int32, device="cuda")
    ops = torch.zeros(q, dtype=torch.uint8, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(3)]
    outs = [torch.zeros(q, dtype=torch.int64, device="cuda") for _ in range(6)]
    torch.cuda.synchronize()
    for k, s in enumerate(streams):
        with torch.cuda.stream(s):
            hs[0].access(dx, outs[k])
            torch.cuda._sleep((k + 1) * SPIN // 2)
            wt.query_multi(hs, zero + (k & 1), ops, zero, dx, outs[3 + k])
    for h in hs:
        h.sync()  # of the build alone
    assert not streams[2].query()
    hs[0].free()
    assert all(s.query() for s in streams)
    hs[1].free()
    for o in outs:
        assert np.array_equal(from_dev_u64(o), S[x].astype(np.uint64))
