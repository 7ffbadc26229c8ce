"""Rank and select at the edges of what one round of loads covers: words,
512-bit blocks, superblocks, and searches between samples over one, a few and
many superblocks, on bitvectors at 16-byte and 8-byte boundaries (Section 5.1
rank and select; every answer against the positions counted on the host)."""
import numpy as np
import pytest

from gpu_util import UMAX, from_dev_u64, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _bits(n, period, seed):
    """n bits, one in `period` set at random (period 0: none)."""
    rng = np.random.default_rng(seed)
    return (rng.integers(0, period, n) == 0) if period else np.zeros(n, bool)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n,period", [(1, 1), (63, 2), (64, 2), (65, 0), (511, 2), (512, 3), (513, 2),
                                      (2047, 2), (2048, 2), (2049, 5), (8192 * 7 + 1, 2),
                                      (1 << 20, 9), ((1 << 22) + 777, 150), (1 << 22, 1000)])
def test_bitvector_rank_select_edges(wt, n, period, offset):
    b = _bits(n, period, n + period)
    words = np.zeros((n + 63) // 64 + offset, np.uint64)
    pad = np.zeros(((n + 63) // 64) * 64, np.uint8)
    pad[:n] = b
    words[offset:] = np.packbits(pad, bitorder="little").view(np.uint64)
    d = to_dev(words)
    h = wt.rs_build(d[offset:], n)
    edges = [e + k for e in (0, 64, 128, 512, 1024, 2048, 4096, 8192, n) for k in (-2, -1, 0, 1)]
    rng = np.random.default_rng(7)
    i = np.unique(np.clip(np.concatenate([edges, rng.integers(0, n, 500)]), 0, n)).astype(np.uint64)
    before = np.concatenate([[0], np.cumsum(b)])
    import torch
    for v in (0, 1):
        out = torch.empty(i.size, dtype=torch.int64, device="cuda")
        h.rank(to_dev(np.full(i.size, v, np.uint32)), to_dev(i), out)
        upto = before[np.minimum(i.astype(np.int64) + 1, n)]
        exp = upto if v else np.minimum(i.astype(np.int64) + 1, n) - upto
        assert np.array_equal(from_dev_u64(out), np.where(i >= n, UMAX, exp.astype(np.uint64)))
        pos = np.flatnonzero(b == bool(v)).astype(np.uint64)
        k = np.unique(np.concatenate([[0, 1, 2, 4096, 4097, 8193, pos.size, pos.size + 1],
                                      rng.integers(1, pos.size + 2, 500)])).astype(np.uint64)
        out = torch.empty(k.size, dtype=torch.int64, device="cuda")
        h.select(to_dev(np.full(k.size, v, np.uint32)), to_dev(k), out)
        ok = (k >= 1) & (k <= pos.size)
        exp = np.full(k.size, UMAX)
        exp[ok] = pos[(k[ok] - 1).astype(np.int64)]
        assert np.array_equal(from_dev_u64(out), exp)
    h.free()


@pytest.mark.parametrize("kind", ["wm", "wt", "huff", "mwt"])
@pytest.mark.parametrize("n,sigma", [(512, 2), (2049, 5), (30011, 300), (300007, 7)])
def test_one_launch_mixes_the_operations(wt, kind, n, sigma):
    """Access, rank and select of one structure side by side in a warp."""
    import torch
    rng = np.random.default_rng(n)
    S = np.minimum(rng.geometric(0.02, n) - 1, sigma - 1).astype(np.uint16)
    build = {"wm": wt.wm_build, "wt": wt.wt_build, "huff": wt.huff_wt_build,
             "mwt": wt.multiary_build}[kind]
    h = build(to_dev(S), sigma)
    q = 700
    op = (np.arange(q) % 3).astype(np.uint8)
    c = rng.integers(0, sigma + 1, q).astype(np.uint32)
    x = rng.integers(0, n + 1, q).astype(np.uint64)
    x[op == 2] %= np.uint64(n // 50 + 2)
    exp = np.full(q, UMAX)
    for t in range(q):
        v, a = int(c[t]), int(x[t])
        if op[t] == 0 and a < n:
            exp[t] = S[a]
        elif op[t] == 1 and a < n and v < sigma:
            exp[t] = np.count_nonzero(S[:a + 1] == v)
        elif op[t] == 2 and v < sigma and a >= 1:
            pos = np.flatnonzero(S == v)
            if a <= pos.size:
                exp[t] = pos[a - 1]
    out = torch.empty(q, dtype=torch.int64, device="cuda")
    wt.query_multi([h], to_dev(np.zeros(q, np.uint32)), to_dev(op), to_dev(c), to_dev(x), out)
    assert np.array_equal(from_dev_u64(out), exp)
    h.free()


@pytest.mark.parametrize("sigma", [2, 3, 256, 300])
@pytest.mark.parametrize("per", [255, 256, 257])
def test_matrix_queries_with_and_without_starts(wt, sigma, per):
    """Rank and select of every symbol (present or not) on both sides of the
    length from which a matrix keeps its symbols' starts."""
    import torch
    L = max(1, (sigma - 1).bit_length())
    n = per << L
    rng = np.random.default_rng(n)
    S = (rng.integers(0, sigma, n) // 2 * 2 % sigma).astype(np.uint16)  # odd symbols absent
    h = wt.wm_build(to_dev(S), sigma)
    c = np.repeat(np.arange(sigma + 1, dtype=np.uint32), 6)
    x = np.tile(np.array([0, 1, n // 3, n - 1, n, per], np.uint64), sigma + 1)
    out = torch.empty(c.size, dtype=torch.int64, device="cuda")
    h.rank(to_dev(c), to_dev(x), out)
    rank = from_dev_u64(out).copy()
    h.select(to_dev(c), to_dev(x), out)
    sel = from_dev_u64(out)
    pos = [np.flatnonzero(S == v) for v in range(sigma + 1)]
    for t in range(c.size):
        v, a = int(c[t]), int(x[t])
        ok = v < sigma and a < n
        assert rank[t] == (np.searchsorted(pos[v], a, side="right") if ok else UMAX)
        ok = v < sigma and 1 <= a <= pos[v].size
        assert sel[t] == (pos[v][a - 1] if ok else UMAX)
    h.free()
