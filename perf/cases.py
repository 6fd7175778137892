"""The calls whose time matters to a program that uses this library, as cases.

A case is a dict of plain values; ``kind`` says which public entry point it
goes through:

* ``extend``    Context.extend            X-drop extension, linear gaps
* ``affine``    Context.extend_affine     the same with affine gaps
* ``matrix``    Context.extend_matrix     letter codes, BLOSUM62, affine gaps
* ``paths``     Context.traceback         alignment paths of the pairs
* ``seeding``   Context.overlap_candidates  k-mer seeding of a read set
* ``overlap``   seeding -> pool -> seeds -> extension -> threshold
* ``serving``   Server.submit / wait      host requests in a mix

Inputs are synthetic, drawn on the GPU from the seed alone, with the length
and error distributions of paper_2002_05200_gb300/synth.py: reads at 5-20 %
error against their source, a share of unrelated pairs that carry one planted
seed, lengths fixed, lognormal, or the heavy-tailed 1 kbp - 1 Mbp mixture.
"""
import math
import os

os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")  # a serving process sets this

import numpy as np
import torch

from paper_2002_05200_gb300 import logan, synth

DEV = "cuda:0"
SEED_LEN = 17
PROTEIN_SEED_LEN = 8


def listed():
    return [
        # a handful of short reads, as a request that came alone: launches and
        # the length of one extension are all it costs
        dict(name="extend_8x2k_ascii", kind="extend", pairs=8, lengths="fixed", median=2000,
             err=0.15, related=1.0, X=50, packed=False, scoring="1,-1,-1"),
        # the small uniform batch: 1,000 pairs of 2 kbp from a parser, ASCII
        dict(name="extend_1k_ascii", kind="extend", pairs=1000, lengths="fixed", median=2000,
             err=0.15, related=1.0, X=50, packed=False, scoring="1,-1,-1"),
        # the headline batch: 100,000 long-read pairs, a fifth unrelated
        dict(name="extend_100k", kind="extend", pairs=100_000, lengths="lognormal", median=10_000,
             err=0.12, related=0.8, X=100, packed=True, scoring="1,-1,-1"),
        # the uneven batch: 1 kbp - 1 Mbp, X of each pair from {10, 50, 100, 500}
        dict(name="extend_uneven_20k", kind="extend", pairs=20_000, lengths="uneven",
             median=1_000_000, err=0.125, related=1.0, X=0, packed=True, scoring="1,-1,-1"),
        # another scoring scheme (gap costlier than a mismatch), ASCII reads
        dict(name="extend_scored_9999", kind="extend", pairs=9_999, lengths="lognormal",
             median=5_000, err=0.10, related=0.9, X=100, packed=False, scoring="2,-3,-5"),
        # affine gaps on long reads
        dict(name="affine_50k", kind="affine", pairs=50_000, lengths="lognormal", median=10_000,
             err=0.12, related=0.8, X=100, packed=True, scoring="1,-1,-2,-1"),
        # protein pairs of a large search and of a small one
        dict(name="matrix_100k", kind="matrix", pairs=100_000, median=450, err=0.25, related=0.8,
             X=60, gaps="-11,-1"),
        dict(name="matrix_1501", kind="matrix", pairs=1_501, median=450, err=0.25, related=0.8,
             X=60, gaps="-11,-1"),
        # the paths of the pairs a caller keeps
        dict(name="paths_10k", kind="paths", pairs=10_000, lengths="lognormal", median=10_000,
             err=0.12, related=0.8, X=100, packed=True, scoring="1,-1,-1"),
        # k-mer seeding of 50,000 reads (10x coverage of a 50 Mbp genome)
        dict(name="seeding_50k", kind="seeding", reads=50_000, mean=10_000, depth=10, k=17,
             min_freq=2, max_freq=4, min_shared=4),
        # the whole many-to-many step of a smaller read set
        dict(name="overlap_8k", kind="overlap", reads=8_000, mean=10_000, depth=10, k=17,
             min_freq=2, max_freq=4, min_shared=4, X=50),
        # a burst of serving requests of mixed sizes, host buffers in and out
        dict(name="serving_24", kind="serving", requests=24, max_pairs=1_000, max_len=1_000_000,
             X=50),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["extend", "extend", "extend", "affine", "matrix", "paths", "seeding",
                       "overlap", "serving"])
    if kind == "matrix":
        return dict(kind=kind, pairs=logu(16, 60_000), median=logu(120, 900),
                    err=round(rng.uniform(0.1, 0.3), 3), related=rng.choice([1.0, 0.8, 0.5]),
                    X=rng.choice([20, 40, 60, 100, 200]), gaps=rng.choice(["-11,-1", "-10,-2", "-9,-1"]))
    if kind in ("seeding", "overlap"):
        c = dict(kind=kind, reads=logu(200, 6_000 if kind == "overlap" else 40_000),
                 mean=logu(2_000, 10_000), depth=rng.choice([5, 10, 15]),
                 k=rng.choice([15, 17, 21]), min_freq=2, max_freq=rng.choice([4, 8]),
                 min_shared=rng.choice([2, 4]))
        if kind == "overlap":
            c["X"] = rng.choice([30, 50, 75])
        return c
    if kind == "serving":
        return dict(kind=kind, requests=rng.randint(1, 24), max_pairs=logu(10, 1_000),
                    max_len=logu(5_000, 1_000_000), X=rng.choice([20, 50, 100]))
    lengths = rng.choice(["fixed", "lognormal", "uneven"])
    X = rng.choice([10, 30, 50, 100, 200, 500] + ([0] if kind == "extend" else []))
    if kind == "paths":
        X = min(X, 200)
    # unrelated pairs keep bands of about 12 X rows under +1/-1/-1
    related = rng.choice([1.0, 0.9, 0.8]) if 0 < X <= 100 and lengths != "uneven" else 1.0
    median = logu(5_000, 400_000) if lengths == "uneven" else logu(150, 20_000)
    mean = 22_000 * min(1.0, median / 300_000) + 2_000 if lengths == "uneven" else median
    # bases x X of a drawn batch stay below a third of the largest listed one's
    most = {"extend": 3e10, "affine": 1.5e10, "paths": 3e9}[kind] / (mean * max(X, 50) * (3 - 2 * related))
    pairs = logu(1, max(2, min(60_000, int(most))))
    scoring = (rng.choice(["1,-1,-2,-1", "1,-1,-4,-1", "2,-3,-5,-2"]) if kind == "affine" else
               rng.choice(["1,-1,-1", "1,-1,-1", "1,-2,-2", "2,-3,-5"]))
    return dict(kind=kind, pairs=pairs, lengths=lengths, median=median,
                err=round(rng.uniform(0.05, 0.18), 3), related=related, X=X,
                packed=rng.random() < 0.7, scoring=scoring)


# ---------------------------------------------------------------------------
# inputs, drawn on the GPU

_CHUNK = 1 << 27  # bases mutated at a time


def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + tag) & 0x7FFFFFFFFFFF)
    return g


def _codes(g, n, K):
    return torch.randint(0, K, (n,), generator=g, device=DEV, dtype=torch.uint8)


def _prefix(x):
    """Exclusive prefix sums of an int64 tensor, one longer than it."""
    return torch.cat([torch.zeros(1, dtype=torch.int64, device=x.device), torch.cumsum(x, 0)])


def _mutate(g, src, rate, protect, types, K):
    """Edit walk: every base outside `protect` suffers an error with
    probability `rate` (a number or one per base): a substitution by another
    letter, an insertion before it, or a deletion, in the shares `types`.
    Returns the output and the output position after each source base."""
    u = torch.rand(src.numel(), generator=g, device=DEV)
    hit = u < rate
    hit[protect] = False
    t = torch.rand(src.numel(), generator=g, device=DEV)
    sub = hit & (t < types[0])
    ins = hit & (t >= types[0]) & (t < types[0] + types[1])
    dele = hit & (t >= types[0] + types[1])
    del u, t, hit
    csum = torch.cumsum(1 + ins.to(torch.int8) - dele.to(torch.int8), 0)
    out = torch.empty(int(csum[-1]) if src.numel() else 0, dtype=torch.uint8, device=DEV)
    val = torch.where(sub, (src + torch.randint(1, K, (src.numel(),), generator=g, device=DEV,
                                                dtype=torch.uint8)) % K, src)
    kept = ~dele
    out[csum[kept] - 1] = val[kept]
    at = csum[ins] - 2
    out[at] = _codes(g, at.numel(), K)
    return out, csum


def _lengths(rng, n, case):
    m = case["median"]
    if case["kind"] == "matrix":  # log-uniform around the median
        x = np.exp(rng.uniform(math.log(m / 4.5), math.log(m * 4.5), size=n))
        return np.maximum(np.rint(x), 2 * PROTEIN_SEED_LEN).astype(np.int64)
    if case["lengths"] == "fixed":
        return np.full(n, m, np.int64)
    if case["lengths"] == "lognormal":
        x = np.rint(rng.lognormal(math.log(m), 0.5, size=n))
        return np.clip(x, max(SEED_LEN, m // 10), 3 * m).astype(np.int64)
    return np.maximum(synth.uneven_lengths(rng, n, m)[0], SEED_LEN).astype(np.int64)


def _pairs(case, seed):
    """Letter codes of both pools, offsets, lengths and seeds of a batch."""
    K, k = (20, PROTEIN_SEED_LEN) if case["kind"] == "matrix" else (4, SEED_LEN)
    n = case["pairs"]
    rng = np.random.default_rng([seed, 11])
    g = _gen(seed, 1)
    n_rel = int(round(case["related"] * n))
    lenA = _lengths(rng, n, case)
    posA = (lenA - k) // 2
    rate = None
    if case["kind"] != "matrix" and case["lengths"] == "uneven":
        rate = torch.from_numpy(rng.uniform(0.4, 1.6, size=n).astype(np.float32) * case["err"]).to(DEV)
    la, pa = torch.from_numpy(lenA).to(DEV), torch.from_numpy(posA).to(DEV)
    offA = _prefix(la)
    poolA = _codes(g, int(offA[-1]), K)
    parts, lens, pos = [], [], []
    cuts = [0]
    ends = np.cumsum(lenA[:n_rel])
    while cuts[-1] < n_rel:  # related pairs: B is A through the edit walk
        done = int(ends[cuts[-1] - 1]) if cuts[-1] else 0
        cuts.append(max(cuts[-1] + 1, int(np.searchsorted(ends, done + _CHUNK, side="right"))))
    for p0, p1 in zip(cuts[:-1], cuts[1:]):
        p1 = min(p1, n_rel)
        b0, b1 = int(offA[p0]), int(offA[p1])
        first = offA[p0:p1] - b0
        prot = (first + pa[p0:p1])[:, None] + torch.arange(k, device=DEV)
        r = case["err"] if rate is None else torch.repeat_interleave(rate[p0:p1], la[p0:p1])
        out, csum = _mutate(g, poolA[b0:b1], r, prot.ravel(), (1 / 3, 1 / 3), K)
        csum = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), csum])
        start = csum[first]
        parts.append(out)
        lens.append(csum[first + la[p0:p1]] - start)
        pos.append(csum[first + pa[p0:p1]] - start)
    if n_rel < n:  # unrelated pairs: an independent B that carries A's seed
        lu = _lengths(rng, n - n_rel, case)
        pu = torch.from_numpy((rng.random(n - n_rel) * (lu - k + 1)).astype(np.int64)).to(DEV)
        lu = torch.from_numpy(lu).to(DEV)
        ou = _prefix(lu)
        b = _codes(g, int(ou[-1]), K)
        t = torch.arange(k, device=DEV)
        b[(ou[:-1] + pu)[:, None] + t] = poolA[(offA[n_rel:n] + pa[n_rel:])[:, None] + t]
        parts.append(b)
        lens.append(lu)
        pos.append(pu)
    poolB, lb, pb = torch.cat(parts), torch.cat(lens), torch.cat(pos)
    offB = _prefix(lb)
    perm = torch.from_numpy(rng.permutation(n)).to(DEV)  # related and unrelated mixed
    seeds = torch.stack([perm, perm, pa[perm], pb[perm], torch.full_like(perm, k)], 1).to(torch.int32)
    Xs = None
    if case["X"] == 0:
        Xs = torch.from_numpy(rng.choice(np.array(synth.UNEVEN_X, np.int32), size=n)).to(DEV)
    return dict(poolA=poolA, offA=offA[:-1].contiguous(), lenA=la, poolB=poolB,
                offB=offB[:-1].contiguous(), lenB=lb, seeds=seeds.contiguous(), Xs=Xs)


def _pack(codes):
    """2-bit words (16 bases a word, one spare word) of a pool of codes."""
    nw = (codes.numel() + 15) // 16
    c = torch.zeros(nw * 16, dtype=torch.uint8, device=DEV)
    c[:codes.numel()] = codes
    q = c.view(-1, 4)
    by = q[:, 0] | (q[:, 1] << 2) | (q[:, 2] << 4) | (q[:, 3] << 6)
    return torch.cat([by, torch.zeros(4, dtype=torch.uint8, device=DEV)]).view(torch.int32)


_ASCII = torch.tensor(list(b"ACGT"), dtype=torch.uint8)


def _pool(codes, off, ln, form):
    if form == "packed":
        bases = _pack(codes)
    else:
        bases = _ASCII.to(DEV)[codes.to(torch.int64)] if form == "ascii" else codes
    return logan.DevicePool(bases, off, ln.to(torch.int32), form == "packed", codes.numel())


def _reads(case, seed):
    """A packed read pool: reads of both strands of one random genome, 12 %
    errors (2 % substitutions, 6 % insertions, 4 % deletions)."""
    rng = np.random.default_rng([seed, 13])
    g = _gen(seed, 2)
    n = case["reads"]
    glen = max(2 * case["mean"], n * case["mean"] // case["depth"])
    genome = _codes(g, glen, 4)
    ln = np.clip(np.rint(rng.lognormal(math.log(case["mean"]) - 0.125, 0.5, size=n)),
                 case["mean"] // 10, glen).astype(np.int64)
    st = (rng.random(n) * (glen - ln + 1)).astype(np.int64)
    rev = torch.from_numpy(rng.random(n) < 0.5).to(DEV)
    ln, st = torch.from_numpy(ln).to(DEV), torch.from_numpy(st).to(DEV)
    parts, lens = [], []
    per = max(1, _CHUNK // (2 * case["mean"]))
    for r0 in range(0, n, per):
        l, s, v = ln[r0:r0 + per], st[r0:r0 + per], rev[r0:r0 + per]
        first = _prefix(l)
        t = torch.arange(int(first[-1]), device=DEV) - torch.repeat_interleave(first[:-1], l)
        vb = torch.repeat_interleave(v, l)
        at = torch.where(vb, torch.repeat_interleave(s + l - 1, l) - t, torch.repeat_interleave(s, l) + t)
        src = genome[at]
        src = torch.where(vb, 3 - src, src)
        out, csum = _mutate(g, src, 0.12, torch.zeros(0, dtype=torch.int64, device=DEV),
                            (2 / 12, 6 / 12), 4)
        csum = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), csum])
        parts.append(out)
        lens.append(csum[first[1:]] - csum[first[:-1]])
    pool, l = torch.cat(parts), torch.cat(lens)
    return _pool(pool, _prefix(l)[:-1].contiguous(), l, "packed")


# ---------------------------------------------------------------------------
# the handles that a program keeps

_held = {}


def _context():
    if "ctx" not in _held:
        _held["ctx"] = logan.Context(0)
    return _held["ctx"]


def _server():
    if "server" not in _held:
        _held["server_ctx"] = logan.Context(0)  # a server uses its context alone
        _held["server"] = logan.Server(_held["server_ctx"], budget_bytes=16 << 30, max_inflight=32)
    return _held["server"]


def _room(rows, *cols, dtype=torch.int32):
    """A program's own buffer for results whose number varies (unused rows 0)."""
    return torch.zeros((rows, *cols), dtype=dtype, device=DEV)


def _into(buf, x):
    n = min(x.shape[0], buf.shape[0])
    buf[:n] = x[:n]
    return buf


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("seeding", "overlap"):
        st["ctx"] = _context()
        st["reads"] = _reads(case, seed)
        n = 6 * case["reads"] * case["depth"]
        st["cands"] = _room(n, 6)
        if kind == "overlap":
            st["results"], st["keep"] = _room(n, 10), _room(n, dtype=torch.uint8)
        return st
    if kind == "serving":
        sizes = synth.request_sizes(np.random.default_rng(case["requests"]), case["requests"],
                                    case["max_pairs"])  # the mix belongs to the case
        p = _pairs(dict(kind="extend", pairs=int(sizes.sum()), lengths="uneven",
                        median=case["max_len"], err=0.125, related=1.0, X=case["X"]), seed)
        sd = p["seeds"].cpu().numpy()
        side = {s: (p["pool" + s].cpu().numpy(), p["off" + s].cpu().numpy(), p["len" + s].cpu().numpy())
                for s in "AB"}
        st["server"], st["requests"], at = _server(), [], 0
        for n in sizes:
            rows = sd[at:at + n]
            at += n
            pools = []
            for s in "AB":
                codes, off, ln = side[s]
                ids = rows[:, 0 if s == "A" else 1]
                own = np.concatenate([codes[off[i]:off[i] + ln[i]] for i in ids])
                pools.append((own, ln[ids]))
            seeds = np.zeros(n, dtype=synth.SEED_DTYPE)
            seeds["idxA"] = seeds["idxB"] = np.arange(n)
            seeds["posA"], seeds["posB"], seeds["len"] = rows[:, 2], rows[:, 3], rows[:, 4]
            w = [synth.pack2bit(synth.ASCII[c]) for c, _ in pools]
            o = [np.concatenate([[0], np.cumsum(l)[:-1]]).astype(np.uint64) for _, l in pools]
            b = synth.Batch("request", w[0], o[0], pools[0][1].astype(np.uint32), w[1], o[1],
                            pools[1][1].astype(np.uint32), seeds, case["X"], packed=True)
            st["requests"].append(logan.HostRequest(b))
        return st
    p = _pairs(case, seed)
    form = "codes" if kind == "matrix" else "packed" if case["packed"] else "ascii"
    st["ctx"] = ctx = _context()
    st["A"] = _pool(p["poolA"], p["offA"], p["lenA"], form)
    st["B"] = _pool(p["poolB"], p["offB"], p["lenB"], form)
    st["seeds"], st["Xs"] = p["seeds"], p["Xs"]
    if kind in ("extend", "affine"):
        st["workspace"] = ctx.workspace(st["A"], st["B"], case["pairs"])
    if kind == "paths":  # codes never outnumber the bases
        st["codes"] = _room(int(min(2.2 * case["pairs"] * case["median"] + 4096, 1.5e8)))
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "extend":
        m, mm, gap = map(int, case["scoring"].split(","))
        return state["ctx"].extend(state["A"], state["B"], state["seeds"], m, mm, gap,
                                   case["X"] or max(synth.UNEVEN_X), state["Xs"],
                                   workspace=state["workspace"])
    if kind == "affine":
        m, mm, go, ge = map(int, case["scoring"].split(","))
        return state["ctx"].extend_affine(state["A"], state["B"], state["seeds"], m, mm, go, ge,
                                          case["X"], workspace=state["workspace"])
    if kind == "matrix":
        go, ge = map(int, case["gaps"].split(","))
        return state["ctx"].extend_matrix(state["A"], state["B"], state["seeds"], synth.BLOSUM62,
                                          go, ge, case["X"])
    if kind == "paths":
        m, mm, gap = map(int, case["scoring"].split(","))
        codes, start, count = state["ctx"].traceback(state["A"], state["B"], state["seeds"], m, mm,
                                                     gap, case["X"])
        # the pairs' codes one after another, without the room between them
        n = count.to(torch.int64)
        first = torch.cumsum(n, 0) - n
        at = torch.repeat_interleave(start - first, n)
        return _into(state["codes"], codes[at + torch.arange(at.numel(), device=at.device)]), count
    if kind == "serving":
        srv = state["server"]
        tickets = [srv.submit(r) for r in state["requests"]]
        for t in tickets:
            status, _ = srv.wait(t)
            if status:
                raise logan.LoganError(status, "request")
        return [r.results for r in state["requests"]]
    ctx, reads = state["ctx"], state["reads"]
    cands = ctx.overlap_candidates(reads, case["k"], case["min_freq"], case["max_freq"],
                                   case["min_shared"])
    if kind == "seeding":
        return _into(state["cands"], cands)
    both = ctx.overlap_pool(reads)
    seeds = ctx.overlap_seeds(cands, reads, case["k"])
    res = ctx.extend(reads, both, seeds, 1, -1, -1, case["X"])
    keep = ctx.overlap_keep(res, seeds, reads, both, 1, 4, 50)
    return (_into(state["cands"], cands), _into(state["results"], res),
            _into(state["keep"], keep))


def work(case):
    """Bytes: pools, seeds and results once.  Operations: integer operations
    of the cells an X-drop sweep evaluates, estimated from the band widths
    that these inputs have (0.85 X rows for reads of one source, about 8 X
    where +1/-1/-1 lets an unrelated pair drift upwards, a third of X for
    protein pairs); 7 a cell with linear gaps, 12 with affine ones."""
    kind = case["kind"]
    if kind in ("seeding", "overlap"):
        bases = case["reads"] * case["mean"]
        cands = 1.3 * case["reads"] * case["depth"]
        b, f = bases / 4 + 24 * cands, 30.0 * bases
        if kind == "overlap":
            b += bases / 4 * 2 + 61 * cands
            f += 7 * 0.85 * case["X"] * cands * case["mean"]
        return {"bytes": b, "flops": f}
    if kind == "serving":
        pairs = case["requests"] * max(1.0, (case["max_pairs"] - 1) / math.log(max(case["max_pairs"], 2)))
        bases = 2 * pairs * (2_000 + 20_000 * min(1.0, case["max_len"] / 300_000))
        return {"bytes": bases / 4 + 60 * pairs, "flops": 7 * 0.85 * case["X"] * bases}
    n = case["pairs"]
    if kind == "matrix":
        bases = 2 * n * case["median"] * 1.4
        return {"bytes": bases + 60 * n, "flops": 12 * case["X"] / 3 * bases}
    if case["lengths"] == "uneven":
        bases = 2 * n * (2_000 + 20_000 * min(1.0, case["median"] / 300_000))
    else:
        bases = 2.2 * n * case["median"]
    X = case["X"] or sum(synth.UNEVEN_X) / len(synth.UNEVEN_X)
    drift = kind != "affine" and case["scoring"] == "1,-1,-1"
    rows = X * (0.85 * case["related"] + (8 if drift else 0.1) * (1 - case["related"]))
    b = bases / (4 if case["packed"] else 1) + 60 * n
    if kind == "paths":
        b += bases * 0.5  # the codes
    return {"bytes": b, "flops": (12 if kind == "affine" else 7) * max(rows, 4) * bases}


# ---------------------------------------------------------------------------
# the extension in plain numpy, 64 bits

_NONE = -(1 << 40)


def _sweep(a, b, sub, go, ge, X):
    """(best, row, column, cells) of one extension of letter codes a, b."""
    m, n = a.size, b.size
    H1, H2, E, F = (np.full(m + 2, _NONE, np.int64) for _ in range(4))  # row i at i + 1
    H1[1] = 0
    lo = hi = best = bi = bj = cells = 0
    for d in range(1, m + n + 1):
        r0, r1 = max(lo, d - n), min(hi + 1, m)
        if r0 > r1:
            break
        cells += r1 - r0 + 1
        i = np.arange(r0, r1 + 1)
        e = np.maximum(E[i + 1] + ge, H1[i + 1] + go + ge)
        f = np.maximum(F[i] + ge, H1[i] + go + ge)
        s = sub[a[np.maximum(i - 1, 0)], b[np.maximum(d - i - 1, 0)]] if m and n else 0
        h = np.maximum(np.maximum(e, f), H2[i] + s)
        live = (h >= best - X) & (h > _NONE // 2)
        rows = np.flatnonzero(live)
        H2, H1 = H1, np.full(m + 2, _NONE, np.int64)
        E, F = np.full(m + 2, _NONE, np.int64), np.full(m + 2, _NONE, np.int64)
        if rows.size == 0:
            break
        at = i[live] + 1
        H1[at], E[at], F[at] = h[live], e[live], f[live]
        lo, hi = r0 + int(rows[0]), r0 + int(rows[-1])
        top = int(h[live].max())
        if top > best:
            best, bi = top, int(i[live][np.argmax(h[live])])
            bj = d - bi
    return best, bi, bj, cells


def exact(case, seed):
    if case["kind"] not in ("extend", "affine", "matrix"):
        return None
    if case["pairs"] * case["median"] * 2.2 > 60_000 or case.get("lengths") == "uneven":
        return None  # (about 50 us an anti-diagonal)
    if case["kind"] == "matrix":
        sub, (go, ge) = synth.BLOSUM62.astype(np.int64), map(int, case["gaps"].split(","))
    else:
        v = list(map(int, case["scoring"].split(",")))
        sub = synth.dna_matrix(v[0], v[1]).astype(np.int64)
        go, ge = (v[2], v[3]) if case["kind"] == "affine" else (0, v[2])
    p = {k: (v.cpu().numpy() if v is not None else None) for k, v in _pairs(case, seed).items()}
    out = np.zeros((case["pairs"], 10), np.int32)
    for r, (ia, ib, pa, pb, k) in enumerate(p["seeds"]):
        a = p["poolA"][p["offA"][ia]:p["offA"][ia] + p["lenA"][ia]]
        b = p["poolB"][p["offB"][ib]:p["offB"][ib] + p["lenB"][ib]]
        X = int(p["Xs"][r]) if p["Xs"] is not None else case["X"]
        L = _sweep(a[:pa][::-1], b[:pb][::-1], sub, go, ge, X)
        R = _sweep(a[pa + k:], b[pb + k:], sub, go, ge, X)
        mid = int(sub[a[pa:pa + k], b[pb:pb + k]].sum())
        out[r, :8] = (L[0] + mid + R[0], L[0], R[0], 0, pa - L[1], pb - L[2], pa + k + R[1],
                      pb + k + R[2])
        out[r, 8:] = np.array([L[3] + R[3]], np.uint64).view(np.int32)
    return torch.from_numpy(out)
