"""The first pass's tile counts and plans: byte alphabets of 2 .. 8 symbols
(counted four bits a symbol), single-pass trees planned from the counts, at
the edges of tiles, of chunks of tiles and of 16-byte alignment; every word
and record against the oracle (integer, tolerance 0)."""
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


@pytest.mark.parametrize("n,offset", [(1, 0), (4095, 1), (4096, 0), (4097, 0), (12288, 3),
                                      (64 * 4096, 0), (64 * 4096 + 1, 0), (400000, 1)])
@pytest.mark.parametrize("sigma", [2, 3, 4, 5, 6, 7, 8, 200])
def test_single_pass_structures(wt, sigma, n, offset):
    rng = np.random.default_rng(sigma * 1000 + n)
    S = rng.integers(0, sigma, n + offset).astype(np.uint8)
    if n > 5000:
        S[offset + 4096:offset + 5000] = sigma - 1
    d = to_dev(S)[offset:]
    S = S[offset:]
    ob, oz = oracle.wm_build(S, sigma)
    h = wt.wm_build(d, sigma)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
    check_binary_dirs(ex, list(ob), [n] * ob.shape[0])
    h.free()
    h = wt.wt_build(d, sigma)
    ex = h.export()
    ot = oracle.wt_build(S, sigma)
    assert np.array_equal(ex.bits.reshape(ot.shape), ot) and np.array_equal(ex.zeros, oz)
    check_binary_dirs(ex, list(ot), [n] * ot.shape[0])
    h.free()
    h = wt.multiary_build(d, sigma)
    ex = h.export()
    om = oracle.mwt_build(S, sigma)
    assert np.array_equal(ex.bits.reshape(om.shape), om)
    h.free()


@pytest.mark.parametrize("sigma", [2, 3, 5, 7, 8])
@pytest.mark.parametrize("n,at", [(4096, 0), (4096, 4095), (5000, 4999), (300000, 77777)])
@pytest.mark.parametrize("bad", [0, 8, 248])
def test_symbol_past_the_alphabet_is_reported(wt, sigma, n, at, bad):
    S = np.random.default_rng(3).integers(0, sigma, n).astype(np.uint8)
    S[at] = sigma + (0 if bad == 0 else bad - sigma if sigma < bad else 0)
    d = to_dev(S)
    for build in (wt.wm_build, wt.wt_build):
        h = build(d, sigma)
        with pytest.raises(wt.WaveletError) as e:
            h.sync()
        assert e.value.status == 2
