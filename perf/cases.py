"""The workloads that users of the library run, as timed cases.

A case is what a program does with one input: a structure built from a
sequence, first queries on it, and its bitmaps and directories handed out as
device arrays; or a batch of queries answered on structures that the program
keeps.  Sizes and
distributions are those of this repository's workloads (2^20 uint8 symbols,
2^30 uint16 Zipf(1.1) symbols, a 2^32-symbol DNA-like text, 2^28 uint32
Zipf(1.0) symbols, 4096 sequences of uneven lengths) and, between them,
ragged sizes of the same ranges.  Inputs are made on the device from the seed.
"""
import ctypes
import math

import numpy as np
import torch

import paper_1610_03524_gb300 as wt

DEV = "cuda"
TORCH_INT = {1: torch.uint8, 2: torch.int16, 4: torch.int32}


def listed():
    return [
        # the smallest call: one short record of a document store
        {"name": "wm_small", "kind": "wm", "n": 5003, "sigma": 200, "width": 1, "zipf": 1.1,
         "queries": 64},
        # an ordinary byte sequence, balanced tree (the 2^20-symbol workload)
        {"name": "wt_1m", "kind": "wt", "n": 1 << 20, "sigma": 256, "width": 1, "zipf": 0.0,
         "queries": 1000},
        # a word-level text: 32-bit ids over a large vocabulary, odd length
        {"name": "wm_12m_u32", "kind": "wm", "n": 12345679, "sigma": 1000003, "width": 4,
         "zipf": 1.0, "queries": 1000},
        # the headline: 2^30 16-bit symbols, 16 levels
        {"name": "wm_1g", "kind": "wm", "n": 1 << 30, "sigma": 1 << 16, "width": 2, "zipf": 1.1,
         "queries": 4096},
        # a sequence handed over in pinned host memory
        {"name": "wm_host", "kind": "wm_host", "n": 50000017, "sigma": 50000, "width": 2,
         "zipf": 1.1, "queries": 4096},
        # genome-like text of 4 letters and a sentinel, balanced tree
        {"name": "wt_genome", "kind": "wt_genome", "n": 1 << 32, "sigma": 5, "width": 1,
         "zipf": 0.0, "queries": 4096},
        # byte text over an odd number of levels, 4-ary tree, then selects on it
        {"name": "mwt_text", "kind": "mwt", "n": 300000007, "sigma": 97, "width": 1, "zipf": 1.0,
         "queries": 1 << 16},
        # Huffman-shaped tree of 2^28 symbols over a 2^20 alphabet
        {"name": "huff_zipf20", "kind": "huff", "n": 1 << 28, "sigma": 1 << 20, "width": 4,
         "zipf": 1.0, "queries": 1 << 16},
        # many sequences of uneven lengths built at once, and queries over them
        {"name": "batch_4096", "kind": "batch", "n": 1 << 31, "seqs": 4096, "queries": 1 << 20},
        # rank queries on the headline's structure
        {"name": "rank_1g", "kind": "rank", "n": 1 << 30, "sigma": 1 << 16, "width": 2,
         "zipf": 1.1, "queries": 1 << 22},
        # the serving loop's step: mixed queries over resident structures
        {"name": "serve_mix", "kind": "serve", "n": 1 << 22, "seqs": 64, "queries": 1 << 16},
        # rank/select directory of a bitvector, odd length
        {"name": "rs_8g", "kind": "rs", "n": (1 << 33) + 12345, "queries": 4096},
    ]


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["wm", "wm", "wm", "wt", "wt", "wm_host", "wt_genome", "mwt", "huff",
                       "batch", "rank", "serve", "rs"])
    few = _log_int(rng, 16, 4096)
    if kind == "rs":
        return {"kind": kind, "n": _log_int(rng, 1000, (1 << 33) + 12345), "queries": few}
    if kind == "batch":
        n = _log_int(rng, 1 << 22, 1 << 31)
        return {"kind": kind, "n": n, "seqs": _log_int(rng, 16, min(4096, n >> 16)),
                "queries": _log_int(rng, 1000, 1 << 20)}
    if kind == "serve":
        return {"kind": kind, "n": _log_int(rng, 1 << 12, 1 << 22), "seqs": _log_int(rng, 2, 64),
                "queries": _log_int(rng, 100, 1 << 16)}
    if kind == "wt_genome":
        return {"kind": kind, "n": _log_int(rng, 1 << 20, 1 << 32), "sigma": 5, "width": 1,
                "zipf": 0.0, "queries": few}
    width = rng.choice([1, 2, 4])
    top = {1: 256, 2: 1 << 16, 4: 1 << 20}[width]
    c = {"kind": kind, "n": _log_int(rng, 1 << 10, {1: 1 << 30, 2: 1 << 30, 4: 1 << 28}[width]),
         "sigma": _log_int(rng, 2, top), "width": width, "zipf": rng.choice([0.0, 1.0, 1.1]),
         "queries": few}
    if kind in ("mwt", "huff"):
        c["n"] = min(c["n"], 1 << 28)
    if kind == "wm_host":
        c["n"] = min(c["n"], 50000017)
    if kind == "rank":
        c["queries"] = _log_int(rng, 100, 1 << 22)
    return c


# ---- inputs ----------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return g


def _symbols(g, n, sigma, width, zipf, out=None):
    """n symbols below sigma: Zipf(zipf) ranks through a random permutation of
    the alphabet, or uniform (zipf = 0)."""
    out = torch.empty(n, dtype=TORCH_INT[width], device=DEV) if out is None else out
    if zipf:
        w = torch.arange(1, sigma + 1, dtype=torch.float64, device=DEV).pow_(-zipf)
        cdf = torch.cumsum(w, 0)
        cdf /= cdf[-1].clone()
        perm = torch.randperm(sigma, generator=g, device=DEV)
    for a in range(0, n, 1 << 27):
        b = min(n, a + (1 << 27))
        if zipf:
            u = torch.rand(b - a, dtype=torch.float64, device=DEV, generator=g)
            r = torch.searchsorted(cdf, u, out_int32=True).clamp_(max=sigma - 1)
            out[a:b] = perm[r].to(out.dtype)
        else:
            out[a:b] = torch.randint(0, sigma, (b - a,), device=DEV, generator=g).to(out.dtype)
    return out


def _genome(g, seed, n):
    """Order-3 Markov text over 0..3 with bursts of mean length 8 (each letter
    repeats with probability 7/8), many chains side by side, and the sentinel 4
    at the end."""
    t = np.random.RandomState(int(seed) % (1 << 31)).gamma(0.5, size=(64, 4)) + 1e-12
    cum = torch.from_numpy(np.cumsum(t / t.sum(1, keepdims=True), 1)[:, :3].astype(np.float32))
    cum = cum.to(DEV)
    steps = 1024 if n >= 1 << 24 else 64
    lanes = (n + steps - 1) // steps
    out = torch.empty((steps, lanes), dtype=torch.uint8, device=DEV)
    ctx = torch.randint(0, 64, (lanes,), device=DEV, generator=g)
    for s in range(steps):
        u = torch.rand(lanes, device=DEV, generator=g)
        new = (u.mul(8.0).frac_().unsqueeze(1) > cum[ctx]).sum(1)
        sym = torch.where(u < 0.125, new, ctx & 3)
        out[s] = sym
        ctx = ((ctx << 2) | sym) & 63
    seq = out.t().reshape(-1)[:n].contiguous()
    seq[-1] = 4
    return seq


def _lengths(rng, m, total):
    """m lengths, log-uniform over [2^10, 2^24], scaled so that they sum to about total."""
    ln = np.exp2(rng.uniform(10, 24, m))
    ln = np.maximum((ln * min(1.0, total / ln.sum())).astype(np.int64), 1 << 10)
    while ln.sum() > total:
        ln[np.argmax(ln)] = max(1 << 10, ln.max() - (ln.sum() - total))
        if ln.max() == 1 << 10:
            break
    return ln


def _mixed_queries(g, ns, sigmas, q):
    """Access, rank and select queries over structures of the given sizes."""
    m = len(ns)
    nd = torch.tensor(ns, dtype=torch.int64, device=DEV)
    sd = torch.tensor(sigmas, dtype=torch.int64, device=DEV)
    sid = torch.randint(0, m, (q,), device=DEV, generator=g)
    op = torch.randint(0, 3, (q,), device=DEV, generator=g)
    r = torch.rand((2, q), dtype=torch.float64, device=DEV, generator=g)
    c = (r[0] * sd[sid]).to(torch.int64)
    span = torch.where(op == 2, nd[sid] // (2 * sd[sid]) + 1, nd[sid])
    x = (r[1] * span).to(torch.int64) + (op == 2)
    return (sid.to(torch.int32), op.to(torch.uint8), c.to(torch.int32), x,
            torch.empty(q, dtype=torch.int64, device=DEV))


def prepare(case, seed):
    g = _gen(seed)
    kind, n = case["kind"], case["n"]
    s = {"kind": kind, "n": n, "sigma": case.get("sigma", 2)}
    if kind == "rs":
        nw = (n + 63) // 64
        bits = torch.randint(-(1 << 63), (1 << 63) - 1, (nw,), device=DEV, generator=g)
        if n & 63:
            bits[-1] &= (1 << (n & 63)) - 1
        s["seq"] = bits
    elif kind == "wt_genome":
        s["seq"] = _genome(g, seed, n)
    elif kind in ("batch", "serve"):
        rng = np.random.RandomState(int(seed) % (1 << 31))
        m = case["seqs"]
        ln = _lengths(rng, m, n) if kind == "batch" else rng.randint(max(1, n // 2), n + 1, m)
        sig = rng.choice([4, 256, 4096, 65536], m)
        zipf = rng.randint(0, 2, m).astype(bool)
        off = np.zeros(m, np.int64)
        flat = torch.empty(int(((ln + 7) // 8 * 8).sum()), dtype=torch.int16, device=DEV)
        at = 0
        for sg in (4, 256, 4096, 65536):
            for z in (False, True):
                begin = at
                for i in np.nonzero((sig == sg) & (zipf == z))[0]:
                    off[i] = at
                    at += (int(ln[i]) + 7) // 8 * 8
                if at > begin:
                    _symbols(g, at - begin, sg, 2, 1.1 if z else 0.0, flat[begin:at])
        s["flat"] = flat
        s["items"] = wt.batch_items(flat.data_ptr(), 2 * off, ln, sig, 2)
        s["m"] = m
        s["q"] = _mixed_queries(g, ln.tolist(), sig.tolist(), case["queries"])
        if kind == "serve":
            s["batch"] = wt.wm_batch_build_one(items=s["items"], ns=m)
            s["handles"] = [s["batch"].handle(i) for i in range(m)]
    else:
        seq = _symbols(g, n, case["sigma"], case["width"], case["zipf"])
        if kind == "wm_host":
            host = torch.empty(seq.shape, dtype=seq.dtype).pin_memory()
            host.copy_(seq)
            seq = host
        s["seq"] = seq
    if kind not in ("batch", "serve"):
        q, sigma = case["queries"], case.get("sigma", 2)
        s["c"] = _symbols(g, q, sigma, 4, case.get("zipf", 0.0))
        s["i"] = torch.randint(0, n, (q,), device=DEV, generator=g)
        s["k"] = torch.randint(1, n // (4 * sigma) + 2, (q,), device=DEV, generator=g)
        s["out"] = torch.empty(q, dtype=torch.int64, device=DEV)
        s["out2"] = torch.empty(q, dtype=torch.int64, device=DEV)
    if kind == "rank":
        s["h"] = wt.wm_build(s.pop("seq"), case["sigma"])
        s["h"].sync()
    return s


# ---- the calls ---------------------------------------------------------------
class _View:
    """A device array of a handle, which it keeps alive."""

    def __init__(self, handle, ptr, count):
        self.handle = handle
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": "<i8", "data": (ptr, False),
                                         "version": 2}


def _array(handle, ptr, count):
    if not count:
        return torch.empty(0, dtype=torch.int64, device=DEV)
    return torch.as_tensor(_View(handle, ptr, count), device=DEV)


def _arrays(h):
    """What the handle holds: level bitmaps, directories and zero counts."""
    v = wt.ExportView()
    st = wt.load_library().wt_export(h.raw, ctypes.byref(v))
    if st != wt.WT_OK:
        raise wt.WaveletError(st, "wt_export")
    L = v.levels
    if v.kind == wt.KIND_HUFF:
        # the lower levels' lengths depend on the code: the root's arrays, which hold every element
        return {"bits": _array(h, v.bits, v.level_off[1]), "dir": _array(h, v.dir, v.dir_off[1]),
                "code_len": np.ctypeslib.as_array(v.code_len, shape=(v.sigma,)).copy(),
                "code": np.ctypeslib.as_array(v.code, shape=(v.sigma,)).copy()}
    out = {"dir": _array(h, v.dir, v.dir_off[L])}
    if v.kind != wt.KIND_RS:
        out["bits"] = _array(h, v.bits, v.level_off[L])
    if v.bits_per_elem == 1:
        out["zeros"] = np.array(v.zeros[:L], dtype=np.int64)
    return out


def _queried(h, s):
    """First queries on a fresh structure: selects (through the samples) and,
    on a Huffman-shaped tree, accesses (through every level)."""
    out = {"select": h.select(s["c"], s["k"], s["out"])}
    if s["kind"] == "huff":
        out["access"] = h.access(s["i"], s["out2"])
    return dict(out, **_arrays(h))


def run(s):
    kind = s["kind"]
    if kind == "wm":
        return _queried(wt.wm_build(s["seq"], s["sigma"]), s)
    if kind == "wm_host":
        return _queried(wt.wm_build_host(s["seq"], s["sigma"]), s)
    if kind in ("wt", "wt_genome"):
        return _queried(wt.wt_build(s["seq"], s["sigma"]), s)
    if kind == "mwt":
        return _queried(wt.multiary_build(s["seq"], s["sigma"]), s)
    if kind == "huff":
        return _queried(wt.huff_wt_build(s["seq"], s["sigma"]), s)
    if kind == "rs":
        return _queried(wt.rs_build(s["seq"], s["n"]), s)
    if kind == "rank":
        return s["h"].rank(s["c"], s["i"], s["out"])
    if kind == "serve":
        return wt.query_multi(s["handles"], *s["q"])
    # batch: build, queue the queries behind it, then read the statuses
    b = wt.wm_batch_build_one(items=s["items"], ns=s["m"])
    answers = wt.query_multi([b.handle(i) for i in range(s["m"])], *s["q"])
    return {"status": b.sync(), "answers": answers}


# ---- accounting and reference --------------------------------------------------
def _levels_of(sigma):
    return max(1, (sigma - 1).bit_length())


def work(case):
    """Input read once, results written once; for queries the arguments, the
    answers and one 64-byte line of bitmap and directory per level and position."""
    kind, n = case["kind"], case["n"]
    per_bit = 1 / 8 + 16 / 2048 + 8 / 4096
    q = case["queries"]
    if kind == "rs":
        return {"bytes": n / 8 + n * (16 / 2048 + 8 / 4096) + q * (20 + 64), "flops": 0}
    if kind in ("batch", "serve"):
        answers = q * (4 + 1 + 4 + 8 + 8) + q * 9.5 * 64
        # 9.5 levels on average over the alphabets 4, 256, 4096 and 65536
        return {"bytes": answers + (n * (2 + 9.5 * per_bit) if kind == "batch" else 0), "flops": 0}
    L = _levels_of(case["sigma"])
    if kind == "rank":
        return {"bytes": q * (4 + 8 + 8 + 2 * 64 * L), "flops": 0}
    if kind == "mwt":
        d = (L + 1) // 2
        return {"bytes": n * (case["width"] + d * (2 / 8 + 64 / 1024 + 8 / 4096))
                + q * (20 + 64 * d), "flops": 0}
    if kind == "huff" and case["zipf"]:
        # a level holds the elements with longer codes: the mean code length, about the entropy
        p = np.arange(1, case["sigma"] + 1, dtype=np.float64) ** -case["zipf"]
        p /= p.sum()
        L = max(1.0, float(-(p * np.log2(p)).sum()))
    return {"bytes": n * (case["width"] + L * per_bit) + q * (20 + 64 * L), "flops": 0}


def _pack(b):
    n = b.numel()
    w = torch.zeros((n + 2047) // 2048 * 2048, dtype=torch.int64, device=DEV)
    w[:n] = b
    return (w.view(-1, 64) << torch.arange(64, device=DEV)).sum(1)


def _directory(b):
    n, nsb = b.numel(), (b.numel() + 2047) // 2048
    z = torch.zeros(nsb * 2048, dtype=torch.int64, device=DEV)
    z[:n] = 1 - b
    blk = z.view(nsb, 4, 512).sum(2)
    rel = torch.cumsum(blk, 1)
    d = torch.zeros((nsb + 1, 2), dtype=torch.int64, device=DEV)
    d[1:, 0] = torch.cumsum(blk.sum(1), 0)
    d[:nsb, 1] = (rel[:, 0] << 16) | (rel[:, 1] << 32) | (rel[:, 2] << 48)
    return d.view(-1)


def _select(seq, sigma, c, k):
    """Positions of the k-th occurrences of c (-1 where there are fewer)."""
    order = torch.sort(seq, stable=True)[1]
    count = torch.bincount(seq, minlength=sigma)
    first = torch.cumsum(count, 0) - count
    c = c.long()
    at = (first[c] + k - 1).clamp(max=seq.numel() - 1)
    return torch.where(k <= count[c], order[at], -1)


def exact(case, seed):
    """The binary structures by their definition: level l's bits are bit
    L-1-l of the symbols in that level's order."""
    if case["kind"] not in ("wm", "wm_host", "wt", "rs") or case["n"] > 1 << 26:
        return None
    s = prepare(case, seed)
    if case["kind"] == "rs":
        b = ((s["seq"].unsqueeze(1) >> torch.arange(64, device=DEV)) & 1).view(-1)[:case["n"]]
        return {"dir": _directory(b), "zeros": np.array([int((b == 0).sum())]),
                "select": _select(b, 2, s["c"], s["k"])}
    seq = s["seq"].to(DEV).to(torch.int64) & ((1 << (8 * case["width"])) - 1)
    L = _levels_of(case["sigma"])
    out = {"dir": [], "bits": [], "zeros": [],
           "select": _select(seq, case["sigma"], s["c"], s["k"])}
    for l in range(L):
        b = (seq >> (L - 1 - l)) & 1
        out["bits"].append(_pack(b))
        out["dir"].append(_directory(b))
        out["zeros"].append(int((b == 0).sum()))
        if case["kind"] == "wt":
            seq = seq[torch.sort(seq >> (L - 1 - l), stable=True)[1]]
        else:
            seq = torch.cat([seq[b == 0], seq[b == 1]])
    return dict(out, dir=torch.cat(out["dir"]), bits=torch.cat(out["bits"]),
                zeros=np.array(out["zeros"]))
