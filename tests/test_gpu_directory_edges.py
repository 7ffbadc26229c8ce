"""Directories at the edges of their groups: levels of one superblock, of one
group of 64 superblocks and of several, levels of different lengths side by
side, and batches of many short sequences (more levels than ride in kernel
parameters); records, totals and samples against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import check_binary_dirs, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


GROUP = 64 * 2048


@pytest.mark.parametrize("n", [0, 1, 2048, 2049, 32 * 2048, 32 * 2048 + 1, GROUP - 1, GROUP,
                               GROUP + 1, 2 * GROUP, 4 * GROUP + 77, 70 * GROUP + 5])
@pytest.mark.parametrize("ones", [0.0, 0.5, 0.003, 1.0])
@pytest.mark.parametrize("offset", [0, 1])
def test_bitvector_directory(wt, n, ones, offset):
    rng = np.random.default_rng(n + int(1000 * ones))
    nw = (n + 63) // 64
    pad = np.zeros(nw * 64, np.uint8)
    pad[:n] = rng.random(n) < ones
    words = np.zeros(nw + offset, np.uint64)
    words[offset:] = np.packbits(pad, bitorder="little").view(np.uint64)
    d = to_dev(words if words.size else np.zeros(1, np.uint64))
    h = wt.rs_build(d[offset:], n)
    ex = h.export()
    level = np.zeros(((n + 2047) // 2048) * 32, np.uint64)
    level[:nw] = words[offset:]
    assert np.array_equal(ex.level_dir(0), oracle.rank_dir(level, n))
    for b in (0, 1):
        assert np.array_equal(ex.samples(0, b), oracle.select_samples(level, n, b))
    h.free()


@pytest.mark.parametrize("n", [70000, GROUP + 3, 700001])
def test_levels_of_different_lengths(wt, n):
    """A Huffman-shaped tree: every level has its own number of groups."""
    rng = np.random.default_rng(n)
    S = np.minimum(rng.geometric(0.3, n) - 1, 40).astype(np.uint8)
    h = wt.huff_wt_build(to_dev(S), 41)
    ex = h.export()
    check_binary_dirs(ex, [ex.level(l) for l in range(ex.levels)], [int(x) for x in ex.level_len])
    h.free()


def test_many_short_levels(wt):
    rng = np.random.default_rng(9)
    ns = [0, 1, 2047, 5000, GROUP - 1, GROUP + 1, 300000] + [int(x) for x in rng.integers(1, 9000, 200)]
    sigmas = [int(x) for x in rng.choice([2, 5, 256, 4096, 65536], len(ns))]
    seqs = [rng.integers(0, s, max(n, 1)).astype(np.uint16) for n, s in zip(ns, sigmas)]
    dev = [to_dev(s) for s in seqs]
    for h, S, n, sigma in zip(wt.wm_batch_build(dev, sigmas, ns=ns), seqs, ns, sigmas):
        ex = h.export()
        ob, oz = oracle.wm_build(S[:n], sigma)
        assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
        check_binary_dirs(ex, list(ob), [n] * ob.shape[0])
        h.free()


@pytest.mark.parametrize("n", [0, 1, 1023, 1025, 32 * 1024 + 1, 64 * 1024 - 1, 64 * 1024,
                               64 * 1024 + 1, 333333, 70 * 64 * 1024 + 9])
@pytest.mark.parametrize("sigma", [2, 4, 77])
def test_digit_directory(wt, n, sigma):
    """Records and samples of every value of every digit level of a 4-ary tree."""
    rng = np.random.default_rng(n + sigma)
    S = np.where(rng.random(n) < 0.6, sigma - 1, rng.integers(0, sigma, n)).astype(np.uint8)
    d = to_dev(S if n else np.zeros(1, np.uint8))
    h = wt.multiary_build(d, sigma, n=n)
    ex = h.export()
    om = oracle.mwt_build(S, sigma)
    assert ex.levels == om.shape[0]
    for b in range(ex.levels):
        assert np.array_equal(ex.level_dir(b), oracle.mwt_dir(om[b], n)), b
        for v in range(4):
            assert np.array_equal(ex.samples(b, v), oracle.digit_samples(om[b], n, v)), (b, v)
    h.free()
