"""Passes whose counting kernel also scans the counts: tile numbers at the
edges of a block (8), of a chunk (64) and of the range (256 chunks) on both
sides, for sequences cut into equal tiles and into the nodes' tiles; every bit
against the oracle (integer, tolerance 0)."""
import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [1, 7, 8, 9, 63, 64, 65, 128, 513, 16383, 16384, 16385])
@pytest.mark.parametrize("short", [0, 1, 2047])
def test_tiles_at_chunk_edges(tiles, short):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as wt
    if tiles > 1000 and short == 2047:
        pytest.skip("as with 1, at a few seconds more")
    n, sigma = tiles * 2048 - short, 20
    S = np.random.default_rng(tiles).integers(0, sigma, n).astype(np.uint8)
    d = to_dev(S)
    ob, oz = oracle.wm_build(S, sigma)
    h = wt.wm_build(d, sigma, tile_symbols=2048)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
    h.free()
    ot = oracle.wt_build(S, sigma)
    h = wt.wt_build(d, sigma)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ot.shape), ot) and np.array_equal(ex.zeros, oz)
    h.free()


def test_chunks_of_more_than_64_tiles():
    """More than 2^20 tiles of 2048 symbols against fewer of 8192 (the same
    bits, whole numbers: equal)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as wt
    n, sigma = (1 << 31) + 4097, 20
    g = torch.Generator(device="cuda").manual_seed(1)
    d = torch.randint(0, sigma, (n,), device="cuda", dtype=torch.uint8, generator=g)
    got = []
    for tile in (2048, 8192):
        h = wt.wm_build(d, sigma, tile_symbols=tile)
        ex = h.export()
        got.append((ex.bits.copy(), ex.zeros.copy()))
        h.free()
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
