"""Device memory that builds hold while they run: the two buffers of the
sequences between the passes are as wide as what is written to each."""
import numpy as np
import pytest

from gpu_util import PoolUse

pytestmark = pytest.mark.gpu

N = 1 << 26
TILE, TAU = 4096, 4


@pytest.fixture(scope="module")
def wt():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1610_03524_gb300 as m
    m.load_library()
    return m


def _symbols(sigma, width):
    import torch
    g = torch.Generator(device="cuda").manual_seed(sigma)
    dt = {1: torch.uint8, 2: torch.int16, 4: torch.int32}[width]
    return torch.randint(0, sigma, (N,), device="cuda", generator=g, dtype=torch.int32).to(dt)


def _buffers(lens):
    """Bytes of the two buffers for levels of the given lengths: pass g writes
    what level 4(g + 1) needs, in 1, 2 or 4 bytes an element, to buffer g & 1."""
    L, b = len(lens), [0, 0]
    for g, a in enumerate(range(TAU, L, TAU)):
        w = 1 if L - a <= 8 else (2 if L - a <= 16 else 4)
        b[g & 1] = max(b[g & 1], int(lens[a]) * w)
    return sum(b)


# tiles' tables (64 bytes of counts and 24 of description, and nodes' tiles),
# directory scratch and class tables, and 2 MB for each allocation's rounding
SLACK = 2 * (N // TILE + (1 << 16)) * 88 + (32 << 20)


@pytest.mark.parametrize("kind,sigma,width", [
    ("wm", 1 << 16, 2), ("wm", 1 << 12, 2), ("wm", 256, 1), ("wm", 1 << 20, 4), ("wm", 1 << 24, 4),
    ("wt", 1 << 16, 2), ("mwt", 1 << 16, 2), ("batch", 1 << 16, 2), ("batch", 1 << 24, 4)])
def test_passes_hold_what_they_write(wt, kind, sigma, width):
    d = _symbols(sigma, width)
    build = {"wm": wt.wm_build, "wt": wt.wt_build, "mwt": wt.multiary_build,
             "batch": lambda x, s: wt.wm_batch_build([x[:N // 2], x[N // 2:]], [s, s])}[kind]
    L = (sigma - 1).bit_length()
    with PoolUse() as use:
        h = build(d, sigma)
    for x in h if kind == "batch" else [h]:
        x.sync()
        x.free()
    assert use.peak <= use.kept + _buffers([N] * L) + SLACK


def test_huffman_passes_hold_what_they_write(wt):
    sigma = 1 << 12
    d = _symbols(sigma, 4)
    d[::2] = 7  # half of the elements have left the tree below the root
    with PoolUse() as use:
        h = wt.huff_wt_build(d, sigma)
        h.sync()
    lens = h.export().level_len
    h.free()
    assert int(lens[TAU]) <= N // 2 + N // 8
    # and the library's copy of the sequence, whose place the codewords take
    assert use.peak <= use.kept + 4 * N + _buffers(lens) + SLACK
    assert np.all(np.diff(lens.astype(np.int64)) <= 0)
