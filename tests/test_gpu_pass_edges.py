"""The partition pass at the edges of its layout: 32-element rows, tiles of
every size, ends of passes of one to four levels, elements of 1, 2 and 4 bytes
at unaligned starts, nodes of a few elements, and symbols so skewed that a tile
has one run; every bit against the oracle (integer, tolerance 0)."""
import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _seq(n, sigma, shape, dtype, seed):
    rng = np.random.default_rng(seed)
    if shape == "uniform":
        S = rng.integers(0, sigma, n)
    elif shape == "skewed":  # nearly all one symbol, the others anywhere
        S = np.where(rng.random(n) < 0.02, rng.integers(0, sigma, n), sigma - 1)
    else:
        S = np.sort(rng.integers(0, sigma, n))
    return S.astype(dtype)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 127, 129, 2047, 2049, 4095, 4096, 4097, 8193,
                               12 * 4096 + 17])
@pytest.mark.parametrize("sigma,dtype", [(2, np.uint8), (9, np.uint8), (256, np.uint8),
                                         (17, np.uint16), (5000, np.uint16), (65536, np.uint16),
                                         (3, np.uint32), (1 << 17, np.uint32)])
@pytest.mark.parametrize("shape", ["uniform", "skewed", "sorted"])
def test_every_structure(wt, n, sigma, dtype, shape):
    offset = n % 3  # starts off the 16-byte boundary too
    S = _seq(n + offset, sigma, shape, dtype, n + sigma)
    d = to_dev(S)[offset:]
    S = S[offset:]
    ob, oz = oracle.wm_build(S, sigma)
    for tile in (2048, 4096, 8192):
        h = wt.wm_build(d, sigma, tile_symbols=tile)
        ex = h.export()
        assert np.array_equal(ex.bits.reshape(ob.shape), ob), tile
        assert np.array_equal(ex.zeros, oz)
        h.free()
    h = wt.wt_build(d, sigma)
    ex = h.export()
    ot = oracle.wt_build(S, sigma)
    assert np.array_equal(ex.bits.reshape(ot.shape), ot) and np.array_equal(ex.zeros, oz)
    h.free()
    h = wt.multiary_build(d, sigma)
    om = oracle.mwt_build(S, sigma)
    assert np.array_equal(h.export().bits.reshape(om.shape), om)
    h.free()
    h = wt.huff_wt_build(d, sigma)
    ex = h.export()
    ln, mx = oracle.huffman_lengths(np.bincount(S, minlength=sigma).astype(np.uint64), 32)
    bits, woff, nl = oracle.huff_wt_build(S, ln, oracle.canonical_codes(ln))
    assert np.array_equal(ex.level_len, nl) and np.array_equal(ex.bits, bits)
    h.free()


@pytest.mark.parametrize("n", [5, 4096, 40001])
def test_batches_of_mixed_widths(wt, n):
    seqs, sigmas = [], []
    for i, (sigma, dtype) in enumerate([(2, np.uint8), (200, np.uint8), (16, np.uint16),
                                        (65536, np.uint16), (1 << 18, np.uint32),
                                        (77, np.uint32)]):
        seqs.append(_seq(n + 7 * i, sigma, "uniform", dtype, i))
        sigmas.append(sigma)
    dev = [to_dev(s) for s in seqs]
    for h, S, sigma in zip(wt.wm_batch_build(dev, sigmas), seqs, sigmas):
        ex = h.export()
        ob, oz = oracle.wm_build(S, sigma)
        assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
        h.free()
