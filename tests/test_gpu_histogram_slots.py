"""Symbol counts of large alphabets through the shared-memory slots: symbols
that share slots, orders in which the slots go to rare symbols first, 16-bit
symbols, ends of the vectors and starts off the 16-byte boundary.  The code
lengths, level lengths and bits that follow from the counts against the oracle
(integer, tolerance 0), and a symbol out of range refused."""
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


N = (1 << 22) + 4099


def _seq(order, sigma, dtype):
    rng = np.random.default_rng(sigma)
    if order == "uniform":
        S = rng.integers(0, sigma, N)
    else:  # a third of it one symbol, another third one of the same slot
        S = rng.integers(0, sigma, N)
        S[rng.random(N) < 0.33] = 5
        S[rng.random(N) < 0.5] = 5 + (1 << 14)
        if order == "rare first":
            hot = (S == 5) | (S == 5 + (1 << 14))
            S = np.concatenate([S[~hot], S[hot]])
        elif order == "falling":
            S = -np.sort(-S)
    return S.astype(dtype)


@pytest.mark.parametrize("sigma,dtype", [(20000, np.uint16), (65536, np.uint16), (70001, np.uint32)])
@pytest.mark.parametrize("order", ["uniform", "mixed", "rare first", "falling"])
@pytest.mark.parametrize("offset", [0, 1])
def test_counts(wt, sigma, dtype, order, offset):
    S = _seq(order, sigma, dtype)
    d = to_dev(S)[offset:]
    S = S[offset:]
    h = wt.huff_wt_build(d, sigma)
    ex = h.export()
    ln, mx = oracle.huffman_lengths(np.bincount(S, minlength=sigma).astype(np.uint64), 32)
    bits, woff, nl = oracle.huff_wt_build(S, ln, oracle.canonical_codes(ln))
    assert np.array_equal(ex.level_len, nl) and np.array_equal(ex.bits, bits)
    h.free()


def test_symbol_out_of_range(wt):
    S = _seq("mixed", 70001, np.uint32)
    S[N - 1] = 70001
    with pytest.raises(wt.WaveletError):
        wt.huff_wt_build(to_dev(S), 70001).sync()
