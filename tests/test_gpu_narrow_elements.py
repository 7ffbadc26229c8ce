"""Alphabets larger than the sequence's elements can hold (1- or 2-byte symbols
under a sigma of more bits): the levels above the elements' width are all
zeros; every bit, zero count and directory against the oracle on the same
values (integer, tolerance 0)."""
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


CASES = [(np.uint8, s) for s in (257, 300, 1025, 5000, 40000, 70000, 1 << 20)] + \
        [(np.uint16, s) for s in (65537, 1 << 18, 1 << 20)]


@pytest.mark.parametrize("dtype,sigma", CASES)
@pytest.mark.parametrize("n", [1, 33, 4097, 50001])
def test_every_structure(wt, dtype, sigma, n):
    rng = np.random.default_rng(n + sigma)
    S = rng.integers(0, np.iinfo(dtype).max + 1, n).astype(dtype)
    d, V = to_dev(S), S.astype(np.uint32)
    ob, oz = oracle.wm_build(V, sigma)
    for tau in (0, 1, 3, 8):
        h = wt.wm_build(d, sigma, tau=tau)
        ex = h.export()
        assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz), tau
        check_binary_dirs(ex, list(ob), [n] * ob.shape[0])
        h.free()
    ot = oracle.wt_build(V, sigma)
    h = wt.wt_build(d, sigma)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ot.shape), ot) and np.array_equal(ex.zeros, oz)
    h.free()
    om = oracle.mwt_build(V, sigma)
    h = wt.multiary_build(d, sigma)
    assert np.array_equal(h.export().bits.reshape(om.shape), om)
    h.free()
    h = wt.huff_wt_build(d, sigma)
    ex = h.export()
    ln, mx = oracle.huffman_lengths(np.bincount(V, minlength=sigma).astype(np.uint64), 32)
    bits, woff, nl = oracle.huff_wt_build(V, ln, oracle.canonical_codes(ln))
    assert np.array_equal(ex.level_len, nl) and np.array_equal(ex.bits, bits)
    h.free()
    for h, in zip(wt.wm_batch_build([d, d], [sigma, sigma])):
        ex = h.export()
        assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
        h.free()


def test_many_bytes_of_a_large_alphabet(wt):
    """Enough of them for the counting of large alphabets."""
    n, sigma = (1 << 22) + 5, 20000
    S = np.random.default_rng(3).integers(0, 256, n).astype(np.uint8)
    h = wt.huff_wt_build(to_dev(S), sigma)
    ex = h.export()
    ln, mx = oracle.huffman_lengths(np.bincount(S, minlength=sigma).astype(np.uint64), 32)
    bits, woff, nl = oracle.huff_wt_build(S, ln, oracle.canonical_codes(ln))
    assert np.array_equal(ex.level_len, nl) and np.array_equal(ex.bits, bits)
    h.free()
