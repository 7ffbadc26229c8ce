"""Trees' passes whose counting kernel also scans the counts: 4096-symbol tiles
and the tiles of the 16 nodes below, whose number the host only bounds, at the
edges of a block (8), of a chunk (64) and of the range (256 chunks) on both
sides.  One symbol alone fills whole tiles of one node, so that the last chunks
that the host's bound allows for are empty.  Every bit and zero count against
the oracle (integer, tolerance 0)."""
import numpy as np
import pytest

import oracle
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

NODES = 16  # of the second pass: five levels, four of them in the first pass
SIGMA, TILE = 20, 4096


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _symbols(n, kind):
    if kind == "one":
        return np.full(n, 13, np.uint8)
    return np.random.default_rng(n).integers(0, SIGMA, n).astype(np.uint8)


def _check(wt, S, multi):
    n, d = S.size, to_dev(S)
    ob = oracle.wt_build(S, SIGMA)
    h = wt.wt_build(d, SIGMA)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ob.shape), ob)
    ones = [int(np.bitwise_count(l).sum()) for l in ob]
    assert ex.zeros.tolist() == [n - k for k in ones]
    h.free()
    if multi:
        om = oracle.mwt_build(S, SIGMA)
        h = wt.multiary_build(d, SIGMA)
        assert np.array_equal(h.export().bits.reshape(om.shape), om)
        h.free()


@pytest.mark.parametrize("kind", ["uniform", "one"])
@pytest.mark.parametrize("short", [0, 1, 4095])
@pytest.mark.parametrize("tiles", [1, 7, 8, 9, 47, 48, 49, 63, 64, 65, 111, 112, 113, 128, 513])
def test_chunk_edges(wt, tiles, short, kind):
    _check(wt, _symbols(tiles * TILE - short, kind), True)


@pytest.mark.parametrize("tiles,kind", [
    (16384 - NODES - 1, "uniform"), (16384 - NODES, "uniform"), (16384 - NODES, "one"),
    (16384 - NODES + 1, "uniform"), (16384, "uniform"), (16384, "one"), (16385, "uniform")])
def test_range_edges(wt, tiles, kind):
    _check(wt, _symbols(tiles * TILE - 1, kind), False)
