"""A build that the device has no memory for says so and leaves nothing behind:
the next call of the thread works."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_dev

pytestmark = pytest.mark.gpu

TOO_MANY = 1 << 39  # symbols of 8 levels: 512 GB of level bits


@pytest.mark.parametrize("kind", ["wm", "wt", "batch", "huff"])
def test_the_next_build_after_one_that_does_not_fit(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as wt
    n, sigma = 10_000, 256
    S = synth.uniform(3, n, sigma, 1)
    d = to_dev(S)
    build = {"wm": wt.wm_build, "wt": wt.wt_build, "huff": wt.huff_wt_build,
             "batch": lambda x, s, n: wt.wm_batch_build([x], [s], ns=[n])}[kind]
    with pytest.raises(wt.WaveletError) as e:
        build(d, sigma, n=TOO_MANY)
    assert e.value.status in ((3, 4) if kind == "huff" else (3,))
    ob, oz = oracle.wm_build(S, sigma)
    h = wt.wm_build(d, sigma)
    ex = h.export()
    assert np.array_equal(ex.bits.reshape(ob.shape), ob) and np.array_equal(ex.zeros, oz)
    h.free()
    t = wt.huff_wt_build(d, sigma)
    t.sync()
    t.free()
    b, = wt.wm_batch_build([d], [sigma])
    b.sync()
    b.free()
