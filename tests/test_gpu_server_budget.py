"""The serving loop's budget covers what a build holds on the device while it
runs, over alphabets of up to 24 bits and elements narrower than the alphabet:
a build is admitted only if its measured peak fits, and one with room to spare
is.  Every structure built this way, alone and in a batch, against the oracle
(integer, tolerance 0)."""
import numpy as np
import pytest

import oracle
from gpu_util import PoolUse, check_binary_dirs, oracle_queries, to_dev

pytestmark = pytest.mark.gpu

NO_MEMORY = 3
FIXED = 16 << 20  # charged to every batch for its tables


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _status(wt, S, sigma, budget):
    srv = wt.Server(budget_bytes=budget)
    try:
        return srv.poll(srv.submit_build(S, sigma))[0]
    finally:
        srv.close()


@pytest.mark.parametrize("dtype,sigma", [
    (np.uint8, 256), (np.uint8, 1 << 16), (np.uint8, 1 << 20), (np.uint16, 5), (np.uint16, 1 << 16),
    (np.uint16, 1 << 22), (np.uint32, 1 << 20), (np.uint32, 1 << 22), (np.uint32, 1 << 24)])
def test_admission_at_the_measured_peak(wt, dtype, sigma):
    n = 1 << 25
    S = np.random.default_rng(sigma).integers(0, min(sigma, np.iinfo(dtype).max + 1), n).astype(dtype)
    with PoolUse() as use:
        assert _status(wt, S, sigma, 1 << 40) == 0
    assert _status(wt, S, sigma, use.peak - 1) == NO_MEMORY
    # one charge for the tables, and their rounding
    assert _status(wt, S, sigma, use.peak + FIXED + (8 << 20)) == 0


CASES = [(np.uint8, 1 << 16), (np.uint8, 1 << 20), (np.uint16, 1 << 22), (np.uint32, 1 << 21),
         (np.uint32, 1 << 22), (np.uint32, 1 << 24), (np.uint16, 300)]


def test_large_alphabets_through_batch_and_server(wt):
    rng = np.random.default_rng(1)
    seqs = [(rng.integers(0, min(s, np.iinfo(t).max + 1), n).astype(t), s)
            for (t, s), n in zip(CASES, (4097, 1, 60001, 33333, 8192, 50000, 12345))]
    for h, (S, s) in zip(wt.wm_batch_build([to_dev(S) for S, _ in seqs], [s for _, s in seqs]), seqs):
        ob, oz = oracle.wm_build(S.astype(np.uint32), s)
        ex = h.export()
        assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
        check_binary_dirs(ex, list(ob), [S.size] * ob.shape[0])
        h.free()
    srv = wt.Server(budget_bytes=1 << 30)
    try:
        ids = [srv.submit_build(S, s) for S, s in seqs]
        for i, (S, s) in zip(ids, seqs):
            q = 999
            x = rng.integers(0, S.size, q).astype(np.uint64)
            op = (np.arange(q) % 3).astype(np.uint8)
            c = S[x].astype(np.uint32)
            x[op == 2] = 1
            st, _, _, out = srv.poll(srv.submit_queries(np.full(q, i, np.uint64), op, c, x), q)
            assert st == 0
            assert np.array_equal(out, oracle_queries(S.astype(np.uint32), s, op, c, x))
    finally:
        srv.close()
