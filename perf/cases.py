"""Timed cases of the search path: what a user of the library has it do, end to end.

A case is one pass through the public entry points (``Index``, ``search``, ``Server``) as a
caller makes it, with every query's ranked alignments read back.  Banks and queries are made
on the GPU from a seed, shaped like the benchmark's synthetic workloads: log-normal sequence
lengths, per-sequence GC, 20 % of the bases in copies of 500 repeat families, a few unknown
bases, queries that are diverged copies of bank regions or random.
"""
import math

import numpy as np
import torch

import paper_1507_02987_gb300 as gn

TINY, MID, LARGE = 1_250_000, 400_000_000, 4_000_000_000  # bank bases
PAPER_MASK = "111010010100110111"


def _case(name, **kw):
    c = dict(name=name, kind="search", bank=MID, nq=1, lo=200, hi=2000, hom=0.5, div=0.25, k=11, stride=11, mask="",
             both=False, w=16, top=100, dist=0, max_e=0.0, device=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one gene-sized query against a bank of 1,000 short sequences
        _case("one_tiny", bank=TINY, nq=1, lo=300, hi=1000, hom=1.0, div=0.06),
        # an interactive query against a genome-scale bank, the plain one-query form
        _case("one_large", bank=LARGE, nq=1, lo=2000, hi=2000, hom=1.0),
        # a query set of uneven lengths, every one a diverged copy, against a mid-size bank
        _case("mid_set", nq=1000, lo=80, hi=10_000, hom=1.0),
        # one call of the command line's full batch (4,096 short queries, half of them unrelated)
        _case("batch_short", nq=4096, lo=50, hi=5000, div=0.30),
        # the band that the autotuner picks for diverged homologs (128 diagonals either side)
        _case("wide_band", nq=1000, lo=50, hi=5000, div=0.30, w=128, device=True),
        # the benchmark's own workload: 2,000 queries against 4 Gbp, queries on the device
        _case("large_set", bank=LARGE, nq=2000, lo=200, hi=20_000, device=True),
        # chromosome-scale queries, cut into segments inside the call
        _case("long_queries", bank=LARGE, nq=8, lo=65_536, hi=1_000_000),
        # the paper's spaced seed, both strands, odd sizes
        _case("mask_strands", nq=333, lo=77, hi=9001, stride=18, mask=PAPER_MASK, both=True),
        # every bank offset indexed: the most sensitive index
        _case("stride_one", nq=500, lo=80, hi=10_000, stride=1, hom=1.0),
        # every alignment under an e-value cut instead of the best hundred
        _case("all_under_e", nq=200, lo=201, hi=5003, top=0, max_e=1e-5),
        # a burst at the request loop over the resident large index
        _case("serve_burst", kind="serve", bank=LARGE, nq=256, lo=50, hi=20_000, hom=0.3),
        # a new bank indexed and searched once, as the console does without a saved index
        _case("index_and_search", kind="build", nq=20, lo=300, hi=3000, device=True),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "set", "set", "wide", "long", "mask", "stride", "all", "serve", "build"])
    bank = _between(rng, TINY, LARGE)
    lo = _between(rng, 50, 400)
    hi = _between(rng, 2 * lo, 20_000)
    c = _case("", bank=bank, lo=lo, hi=hi, hom=rng.choice([0.3, 0.5, 1.0]), div=rng.choice([0.06, 0.25, 0.30]),
              device=rng.random() < 0.3)
    if kind == "one":
        c.update(nq=_between(rng, 1, 12), hom=1.0)
    elif kind == "set":
        c.update(nq=_between(rng, 13, 2000), k=rng.choice([11, 11, 12]), dist=rng.choice([0, 0, 22, 66]))
        c["stride"] = c["k"]
    elif kind == "wide":
        c.update(bank=min(bank, MID), nq=_between(rng, 10, 800), hi=min(hi, 5000), w=rng.choice([32, 64, 100, 128]))
    elif kind == "long":
        c.update(nq=_between(rng, 1, 8), lo=65_536, hi=_between(rng, 70_000, 1_000_000))
    elif kind == "mask":
        c.update(bank=min(bank, MID), nq=_between(rng, 10, 400), stride=rng.choice([18, 9]), mask=PAPER_MASK,
                 both=rng.random() < 0.5)
    elif kind == "stride":
        c.update(bank=min(bank, MID), nq=_between(rng, 10, 500), hi=min(hi, 10_000), stride=rng.choice([1, 1, 4]))
    elif kind == "all":
        c.update(bank=min(bank, MID), nq=_between(rng, 5, 200), hi=min(hi, 5000), top=0, max_e=rng.choice([1e-5, 1e-20]))
    elif kind == "serve":
        c.update(kind="serve", nq=_between(rng, 16, 256), device=False)
    else:
        c.update(kind="build", bank=min(bank, MID), nq=_between(rng, 1, 20), stride=rng.choice([11, 4]), device=True)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs --
def _letters(gc, bit):  # A, T or C, G
    return 65 + 2 * gc + bit * (19 - 15 * gc)


def _random_bases(n, g):
    r = torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda", generator=g)
    return _letters(r & 1, r >> 1)


def _flat(lens):
    """(row, offset in row) of every element of rows of the given lengths."""
    row = torch.repeat_interleave(torch.arange(len(lens), device="cuda"), lens)
    return row, torch.arange(len(row), device="cuda") - (torch.cumsum(lens, 0) - lens)[row]


def _bank(n_bases, seed):
    """Sequence starts (host) and ASCII bases (GPU) of a bank of about n_bases bases."""
    rng = np.random.default_rng([seed, 1])
    g = torch.Generator("cuda").manual_seed(seed)
    small = n_bases <= 2 * TINY
    if small:
        lens = rng.integers(500, 2001, max(1, n_bases // 1250))
    else:
        med, top = (1200.0, 200_000) if n_bases > MID else (1500.0, 50_000)
        lens = np.exp(rng.normal(math.log(med), 0.7585, max(1, int(n_bases / (1.333 * med))))).astype(np.int64)
        lens = np.clip(lens, 100, top)
    start = np.zeros(len(lens) + 1, np.uint64)
    start[1:] = np.cumsum(lens)
    n = int(start[-1])
    bases = torch.empty(n, dtype=torch.uint8, device="cuda")
    dev_lens = torch.from_numpy(np.ascontiguousarray(lens)).cuda()
    share = (0.35 + 0.30 * torch.rand(len(lens), device="cuda", generator=g)) * (0 if small else 1) + (0.5 if small else 0)
    gc = (share * 256).to(torch.uint8)
    cuts = np.unique(np.append(np.searchsorted(start, np.arange(0, n, 1 << 27)), len(lens)))
    for a, b in zip(cuts[:-1], cuts[1:]):
        x, y = int(start[a]), int(start[b])
        r = torch.randint(0, 256, (y - x,), dtype=torch.uint8, device="cuda", generator=g)
        bit = torch.randint(0, 2, (y - x,), dtype=torch.uint8, device="cuda", generator=g)
        bases[x:y] = _letters((r < torch.repeat_interleave(gc[a:b], dev_lens[a:b], output_size=y - x)).to(torch.uint8), bit)
    if not small:
        # copies of 500 families at 1-10 % divergence over a fifth of the bases, one to a slot
        fam = np.exp(rng.uniform(math.log(300), math.log(6000), 500)).astype(np.int64)
        cons = _random_bases(int(fam.sum()), g)
        slot = int(5 * fam.mean())
        at = torch.from_numpy(np.concatenate([[0], np.cumsum(fam)[:-1]])).cuda()
        fam = torch.from_numpy(fam).cuda()
        for s0 in range(0, n // slot, 32768):
            m = min(32768, n // slot - s0)
            f = torch.randint(0, 500, (m,), device="cuda", generator=g)
            to = (s0 + torch.arange(m, device="cuda")) * slot + (
                torch.rand(m, device="cuda", generator=g) * (slot - fam[f]).clamp(min=0)).long()
            ln = torch.minimum(fam[f], n - to)
            row, off = _flat(ln)
            div = 0.01 + 0.09 * torch.rand(m, device="cuda", generator=g)
            v = cons[at[f][row] + off]
            hit = torch.rand(len(v), device="cuda", generator=g) < div[row]
            v = torch.where(hit, _random_bases(len(v), g), v)
            bases[to[row] + off] = v
    bases[torch.randint(0, n, (n // 100_000,), device="cuda", generator=g)] = ord("N")
    return start, bases


def _queries(c, start, bases, seed):
    """Query starts (host) and bases (GPU): diverged copies of bank regions (substitutions and
    single-base indels, 5 to 1), the others random."""
    rng = np.random.default_rng([seed, 2])
    g = torch.Generator("cuda").manual_seed(seed + 1)
    nq = c["nq"]
    lens = np.exp(rng.uniform(math.log(c["lo"]), math.log(c["hi"]), nq)).round().astype(np.int64)
    hom = rng.random(nq) < c["hom"]
    slen = np.diff(start.astype(np.int64))
    by_len = np.argsort(-slen, kind="stable")
    div = rng.uniform(0.02 if c["div"] > 0.1 else c["div"], c["div"], nq)
    hom[0], div[0], lens[0] = True, div[0] / 3, max(lens[0], min(200, c["hi"]))  # one that is surely found
    enough = np.searchsorted(-slen[by_len], -lens, side="right")
    src = by_len[(rng.random(nq) * np.maximum(enough, 1)).astype(np.int64)]
    part = np.where(hom, np.minimum(lens, slen[src]), 0)  # the part that is copied
    pos = start[src].astype(np.int64) + (rng.random(nq) * (slen[src] - part + 1)).astype(np.int64)
    row, off = _flat(torch.from_numpy(lens).cuda())
    copy = off < torch.from_numpy(part).cuda()[row]
    tdiv = torch.from_numpy(div).cuda()[row] * copy
    copied = bases[torch.from_numpy(pos).cuda()[row] * copy + off * copy]
    v = torch.where(copy, copied, _random_bases(len(row), g))
    v = torch.where(torch.rand(len(v), device="cuda", generator=g) < tdiv * 5 / 6, _random_bases(len(v), g), v)
    r = torch.rand(len(v), device="cuda", generator=g)
    gone, more = r < tdiv / 12, (r >= tdiv / 12) & (r < tdiv / 6)
    rep = torch.ones_like(row) - gone.long() + more.long()
    out = torch.repeat_interleave(v, rep)
    end = torch.cumsum(rep, 0)
    out[end[more] - 1] = _random_bases(int(more.sum()), g)
    qstart = np.zeros(nq + 1, np.uint64)
    qstart[1:] = end[torch.from_numpy(np.cumsum(lens) - 1).cuda()].cpu().numpy()
    return qstart, out


def prepare(case, seed):
    c = dict(case)
    start, bases = _bank(c["bank"], seed)
    qstart, qbases = _queries(c, start, bases, seed)
    s = {"case": c, "qstart": qstart, "qbases": qbases if c["device"] else qbases.cpu().numpy()}
    s["params"] = gn.make_params(max_hit_distance=c["dist"], max_alignments=c["top"], band_w=c["w"],
                                 max_evalue=c["max_e"] or math.inf,
                                 flags=gn.GN_FLAG_BOTH_STRANDS if c["both"] else 0)
    # the caller's result table: room for every alignment a call can return
    rows = c["nq"] * (2 if c["both"] else 1) * (c["top"] or 4096)
    s["table"] = {f: np.zeros(rows, gn.HIT_DTYPE[f]) for f in gn.HIT_DTYPE.names if f != "query"}
    s["rows"] = 0
    if c["kind"] == "build":
        s.update(start=start, bases=bases)
        return s
    s["index"] = gn.Index(start, bases, k=c["k"], stride=c["stride"], mask=c["mask"] or None)
    if c["kind"] == "serve":
        s["server"] = gn.Server(s["index"], 16 << 30, params=s["params"])
        s["requests"] = [s["qbases"][int(a):int(b)].tobytes() for a, b in zip(qstart[:-1], qstart[1:])]
    return s


def _into_table(s, per_query):
    hits = np.concatenate(per_query)
    for f, col in s["table"].items():
        col[:len(hits)] = hits[f]
        col[len(hits):s["rows"]] = 0
    s["rows"] = len(hits)
    return dict(s["table"], counts=np.array([len(h) for h in per_query]))


def _search(s, index):
    res = gn.search(index, s["qstart"], s["qbases"], params=s["params"])
    hits = res.all()
    res.close()
    return _into_table(s, hits)


def run(s):
    kind = s["case"]["kind"]
    if kind == "search":
        return _search(s, s["index"])
    if kind == "build":
        index = gn.Index(s["start"], s["bases"], k=s["case"]["k"], stride=s["case"]["stride"])
        out = _search(s, index)
        index.close()
        return out
    tickets = [s["server"].submit(q) for q in s["requests"]]
    hits = []
    for t in tickets:
        res = s["server"].poll(t)
        hits.append(res.query(0))
        res.close()
    return _into_table(s, hits)


def work(case):
    c = case
    m = c["nq"] * (c["hi"] - c["lo"]) / max(math.log(c["hi"] / c["lo"]), 1e-9) if c["hi"] > c["lo"] else c["nq"] * c["lo"]
    m *= 2 if c["both"] else 1
    k = c["mask"].count("1") if c["mask"] else c["k"]
    windows = c["bank"] / c["stride"]
    hits = m * windows / 4 ** k            # one 4-byte occurrence each
    aln = c["nq"] * (2 if c["both"] else 1) * min(24.0, 2.0 + hits / m)
    nbytes = m + 8.0 * min(m, 4 ** k) + 4.0 * hits + 48.0 * aln
    ops = 8.0 * aln * 190 * (2 * c["w"] + 2)  # banded alignment: 8 integer operations a cell
    if c["kind"] == "build":
        nbytes += 1.375 * c["bank"] + 4.0 * windows + 8.0 * 4 ** k
    return {"bytes": nbytes, "flops": ops}


# ------------------------------------------------------------------- exact --
def _extend(q, d, qi, di, step):
    best = score = ext = e = 0
    while 0 <= qi < len(q) and 0 <= di < len(d):
        e += 1
        score += 1 if q[qi] == d[di] and q[qi] in b"ACGT" else -3
        if score > best:
            best, ext = score, e
        elif best - score > 20:
            break
        qi, di = qi + step, di + step
    return ext


def _align(q, d, h, w):
    """Banded affine-gap local alignment around a box: score and ranges (ties: the diagonal
    before a gap, opening before extending, the first cell of the highest score)."""
    qs, qe, ds, de = h
    lo, hi = min(ds - qs, de - qe) - w, max(ds - qs, de - qe) + w
    i0, i1, j0, j1 = max(0, qs - w), min(len(q), qe + w), max(0, ds - w), min(len(d), de + w)
    none, best, prev = (-1 << 29, None), (0,), {}
    for i in range(i0, i1):
        row, fv, left = {}, none, None
        for j in range(max(j0, i + lo), min(j1 - 1, i + hi) + 1):
            up, dg = prev.get(j), prev.get(j - 1)
            e = none
            if up:
                e = (up[0][0] - 7, up[0][1]) if up[0][0] - 7 >= up[1][0] - 2 else (up[1][0] - 2, up[1][1])
            if left:
                fv = (left[0] - 7, left[1]) if left[0] - 7 >= fv[0] - 2 else (fv[0] - 2, fv[1])
            b = dg[0] if dg and dg[0][0] > 0 else (0, (i, j))
            c = (b[0] + (1 if q[i] == d[j] and q[i] in b"ACGT" else -3), b[1])
            if e[0] > c[0]:
                c = e
            h0 = (max(c[0], 0), c[1])
            left = h0
            cell = h0 if h0[0] >= fv[0] else fv
            if cell[0] > best[0]:
                best = (cell[0], cell[1], i, j)
            row[j] = (cell, e)
        prev = row
    return (best[0], best[1][0], best[2] + 1, best[1][1], best[3] + 1) if best[0] else None


def exact(case, seed):
    """The method step by step on the host, for one query against the smallest banks; larger
    cases would take minutes."""
    c = case
    if c["kind"] != "search" or c["bank"] > 2 * TINY or c["nq"] * c["hi"] > 2000 or c["stride"] != 11 or c["mask"]:
        return None
    start, bases = _bank(c["bank"], seed)
    qstart, qb = _queries(c, start, bases, seed)
    bases, qb = bases.cpu().numpy().tobytes(), qb.cpu().numpy().tobytes()
    start, k, t, w = [int(x) for x in start], c["k"], c["stride"], c["w"]
    dist, table = c["dist"] or 3 * t, {}
    for s in range(len(start) - 1):
        for g in range(start[s], start[s + 1] - k + 1, t):
            table.setdefault(bases[g:g + k], []).append((s, g - start[s]))
    ranked = []
    for n in range(c["nq"]):
        q = qb[int(qstart[n]):int(qstart[n + 1])]
        diag = {}
        for x in range(len(q) - k + 1):
            if b"N" not in q[x:x + k]:
                for s, p in table.get(q[x:x + k], ()):
                    diag.setdefault((s, p - x), []).append(x)
        boxes = {}
        for (s, dg), xs in diag.items():
            ends = [i for i in range(len(xs)) if i + 1 == len(xs) or xs[i + 1] - xs[i] > dist]
            for a, b in zip([0] + [i + 1 for i in ends[:-1]], ends):
                qs, qe = xs[a], xs[b] + k
                if qe - qs >= 2 * k:
                    d = bases[start[s]:start[s + 1]]
                    el, er = _extend(q, d, qs - 1, qs + dg - 1, -1), _extend(q, d, qe, qe + dg, 1)
                    boxes.setdefault(s, []).append((qs - el, qs + dg - el, qe + er, qe + dg + er))
        merged = []
        for s, hs in boxes.items():
            hs.sort()
            cur = None
            for qs, ds, qe, de in hs:
                if cur and qs < cur[2] and cur[0] < qe and ds < cur[3] and cur[1] < de:
                    cur = (min(cur[0], qs), min(cur[1], ds), max(cur[2], qe), max(cur[3], de))
                else:
                    merged += [(s,) + cur] if cur else []
                    cur = (qs, ds, qe, de)
            merged.append((s,) + cur)
        merged.sort(key=lambda m: (-min(m[3] - m[1], m[4] - m[2]), m))
        best = {}
        for s, qs, ds, qe, de in merged[:c["top"] or None]:
            a = _align(q, bases[start[s]:start[s + 1]], (qs, qe, ds, de), w)
            if a:
                key = (s,) + a[1:]
                best[key] = max(best.get(key, 0), a[0])
        rows = sorted(((sc,) + key for key, sc in best.items()), key=lambda r: (-r[0], r[1], r[2], r[4], r[3], r[5]))
        ev = [(0.711 * len(q) * start[-1] * math.exp(-1.3740631 * r[0])) for r in rows]
        ranked.append([(*r, i, e) for i, (r, e) in enumerate(zip(rows, ev)) if e <= (c["max_e"] or math.inf)])
    flat = [r + ((1.3740631 * r[0] - math.log(0.711)) / math.log(2.0),) for rows in ranked for r in rows]
    cols = {f: np.zeros(c["nq"] * (c["top"] or 4096), np.float64 if f in ("evalue", "bits") else np.int64)
            for f in ("score", "seq", "q_start", "q_end", "db_start", "db_end", "rank", "evalue", "bits")}
    for i, r in enumerate(flat):
        for f, x in zip(cols, r):
            cols[f][i] = x
    return dict(cols, counts=np.array([len(r) for r in ranked]))
