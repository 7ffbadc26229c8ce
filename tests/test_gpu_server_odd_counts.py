"""Query requests of any number of queries through the serving loop: its staging
buffer holds arrays of 4, 1, 4 and 8 bytes a query one after another, and the
8-byte ones are read as such whatever the count."""
import numpy as np
import pytest

import synth
from gpu_util import oracle_queries

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [[1], [3], [7], [8], [999], [1000, 1], [5, 2, 4], [65537]])
def test_any_number_of_queries(counts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as wt
    n, sigma = 20000, 300
    S = synth.zipf(11, n, sigma, 1.1, 2)
    srv = wt.Server(budget_bytes=1 << 30)
    try:
        i = srv.submit_build(S, sigma)
        qs = [synth.queries(20 + k, S, sigma, q) for k, q in enumerate(counts)]
        reqs = [srv.submit_queries(np.full(op.size, i, np.uint64), op, c, x) for op, c, x in qs]
        for r, (op, c, x) in zip(reqs, qs):
            st, _, _, out = srv.poll(r, op.size)
            assert st == 0
            assert np.array_equal(out, oracle_queries(S, sigma, op, c, x))
    finally:
        srv.close()
