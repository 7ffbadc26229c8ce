"""Huffman codes of large alphabets, built on the device: lengths, codes, node
tables (through the bitmaps and queries), zero counts and directories equal the
oracle's heap merge, on uniform, Zipf-like and equal weights, with absent
symbols, on weights whose code is longer than 32 bits (left to the host), and
at both sides of the alphabet size that decides who builds it."""
import numpy as np
import pytest

import oracle
from gpu_util import check_binary_dirs, from_dev_u64, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _sequence(kind, sigma, n, rng):
    if kind == "uniform":
        return rng.integers(0, sigma, n)
    if kind == "equal":  # every present symbol as often as the others
        return np.resize(rng.permutation(sigma)[:max(1, sigma // 3)], n)
    if kind == "one":
        return np.full(n, sigma - 1)
    if kind == "two":
        return np.where(np.arange(n) % 7 == 0, 5, sigma - 2)
    if kind == "zipf":
        w = np.arange(1, sigma + 1) ** -1.0
        return rng.permutation(sigma)[np.searchsorted(np.cumsum(w / w.sum()), rng.random(n)).clip(0, sigma - 1)]
    # weights 1, 1, 2, 3, 5, ...: one symbol per length
    f = [1, 1]
    while sum(f) + f[-1] + f[-2] <= n:
        f.append(f[-1] + f[-2])
    return rng.permutation(np.repeat(np.arange(len(f)) * (sigma // 64), f))


@pytest.mark.parametrize("sigma", [65535, 65536, 65537, 200000])
@pytest.mark.parametrize("kind,n", [("uniform", 300000), ("uniform", 1000), ("equal", 250001),
                                    ("one", 5000), ("two", 5000), ("zipf", 400000),
                                    ("fibonacci", 60000), ("fibonacci", 20000000)])
def test_codes_equal_the_oracle(wt, sigma, kind, n):
    if kind == "fibonacci" and n > 100000 and sigma != 65536:
        pytest.skip("one alphabet is enough for the long code")
    rng = np.random.default_rng(sigma + n)
    S = np.ascontiguousarray(_sequence(kind, sigma, n, rng).astype(np.uint32))
    n = S.size
    h = wt.huff_wt_build(to_dev(S), sigma)
    ex = h.export()
    hist = np.bincount(S, minlength=sigma).astype(np.uint64)
    ln, mx = oracle.huffman_lengths(hist, 32)
    code = oracle.canonical_codes(ln)
    assert ex.max_code_len == mx
    assert np.array_equal(ex.code_len, ln) and np.array_equal(ex.code, code)
    if n <= 400001:
        bits, woff, nl = oracle.huff_wt_build(S, ln, code)
        assert np.array_equal(ex.level_len, nl) and np.array_equal(ex.level_off, woff)
        assert np.array_equal(ex.bits, bits)
        check_binary_dirs(ex, [ex.level(l) for l in range(mx)], [int(x) for x in nl])
    import torch
    i = rng.integers(0, n, 3000).astype(np.uint64)
    out = torch.empty(i.size, dtype=torch.int64, device="cuda")
    h.access(to_dev(i), out)
    assert np.array_equal(from_dev_u64(out), S[i.astype(np.int64)].astype(np.uint64))
    h.free()


def test_bad_symbol_is_reported(wt):
    S = np.arange(100000, dtype=np.uint32) % 70000
    h = wt.huff_wt_build(to_dev(S), 69999)
    with pytest.raises(wt.WaveletError) as e:
        h.sync()
    assert e.value.status == 2
