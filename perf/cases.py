"""The work that users have the signature join do, as measurable cases.

Every case goes through the package's public calls on relations that are
resident on the GPU.  Sizes and key lengths are those of the workloads in
`workloads/` and `bench.py` (plain, large, medium, collision, batch and
serving), at their full or profiling size.

A join returns its pairs in no particular order.  R's keys are distinct in
these cases (a lookup of S rows in a keyed R), so each program here goes on
as such a user's does: it writes the pairs into a column that holds, for every
S row, its R row or -1.  That column has one value for given inputs.
"""
import math
import random

import torch

import paper_2411_18183_gb300 as ag

DEV = "cuda"
CHUNK = 1 << 27                    # bytes handled at once while inputs are made

BATCH_BANDS = ((32, 128), (256, 1024), (2048, 8192))


def listed():
    return [
        # a handful of keys signed for a lookup: launch and latency count
        {"name": "sig_tiny", "op": "sig", "n": 1000, "lo": 32, "hi": 128, "text": "printable", "ncomp": 4},
        # many short keys (names, codes, URLs): the work per key counts
        {"name": "sig_short", "op": "sig", "n": 4_000_000, "lo": 32, "hi": 128, "text": "printable", "ncomp": 4},
        # a relation of text keys, larger than the L2 cache: the common bulk call
        {"name": "sig_mid", "op": "sig", "n": 2_000_000, "lo": 256, "hi": 1024, "text": "printable", "ncomp": 4},
        # the paper's two-symbol signature over long DNA-like keys
        {"name": "sig_two_long", "op": "sig", "n": 300_000, "lo": 2048, "hi": 8192, "text": "acgt", "ncomp": 2},
        # the paper's byte-symbol signature over markup-like keys
        {"name": "sig_bytes", "op": "gf8", "n": 1_000_000, "lo": 200, "hi": 2000, "text": "alnum"},
        # cumulative signatures at 256-byte blocks, for later substring lookups
        {"name": "sig_prefixes", "op": "prefixes", "n": 500_000, "lo": 200, "hi": 2000, "text": "alnum", "block": 256},
        # the small whole join, in one convenience call (buffers allocated by the call)
        {"name": "join_plain", "op": "join", "m": 10_000, "n": 100_000, "lo": 64, "hi": 256, "text": "printable",
         "copy": 0.30, "near": 0.0, "zipf": 0.0, "call": "join"},
        # the large whole join with skewed partners, buffers kept by the caller
        {"name": "join_large", "op": "join", "m": 1_000_000, "n": 10_000_000, "lo": 256, "hi": 1024,
         "text": "printable", "copy": 0.50, "near": 0.0, "zipf": 1.1, "call": "into"},
        # long keys, most of them equal or nearly equal to an R key
        {"name": "join_near", "op": "join", "m": 100_000, "n": 1_000_000, "lo": 2048, "hi": 8192, "text": "acgt",
         "copy": 0.40, "near": 0.40, "zipf": 0.0, "call": "into"},
        # the join on the keys' first 256 bytes
        {"name": "join_prefix", "op": "join", "m": 200_000, "n": 2_000_000, "lo": 256, "hi": 1024,
         "text": "printable", "copy": 0.50, "near": 0.0, "zipf": 0.0, "call": "prefix", "prefix": 256},
        # many independent joins of uneven sizes and key lengths in one prepared batch
        {"name": "join_batch", "op": "batch", "joins": 24, "median": 5_000, "factor": 10, "text": "printable",
         "copy": 0.25, "gaps": False},
        # a table that a serving process keeps, probed by one query for the rows with a partner; signatures returned
        {"name": "probe_semi", "op": "probe", "m": 50_000, "n": 500_000, "lo": 200, "hi": 2000, "text": "alnum",
         "copy": 0.20, "near": 0.0, "zipf": 0.0, "call": "semi"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sig", "sig", "gf8", "prefixes", "join", "join", "join", "batch", "probe", "probe"])
    text = rng.choice(["printable", "acgt", "alnum"])
    if op == "batch":
        return {"op": op, "joins": _log(rng, 2, 24), "median": _log(rng, 1000, 5_000), "factor": rng.randint(4, 16),
                "text": text, "copy": round(rng.uniform(0.1, 0.5), 3), "gaps": rng.random() < 0.5}
    lo = _log(rng, 32 if text == "acgt" else 16, 2048)       # long enough for R's keys to be distinct
    hi = min(8192, lo * rng.randint(1, 8) + rng.randint(0, 31))
    most = 1e9 if op in ("gf8", "prefixes") else 3e9
    n = max(500, int(_log(rng, 5e4, most) / (0.5 * (lo + hi) + 24)))
    if op == "sig":
        return {"op": op, "n": n, "lo": lo, "hi": hi, "text": text, "ncomp": rng.choice([4, 4, 2])}
    if op == "gf8":
        return {"op": op, "n": n, "lo": lo, "hi": hi, "text": text}
    if op == "prefixes":
        return {"op": op, "n": n, "lo": lo, "hi": hi, "text": text, "block": rng.choice([16, 32, 64, 256, 256, 1024, 4096])}
    case = {"op": op, "m": max(50, n // rng.randint(2, 16)), "n": n, "lo": lo, "hi": hi, "text": text,
            "copy": round(rng.uniform(0.05, 0.6), 3), "near": round(rng.choice([0.0, 0.0, rng.uniform(0.05, 0.4)]), 3),
            "zipf": rng.choice([0.0, 0.0, 1.1])}
    if op == "probe":
        case["call"] = rng.choice(["inner", "inner", "semi", "anti", "semi_r", "anti_r"])
    else:
        case["call"] = rng.choice(["join", "into", "into", "prefix", "partitioned"])
        if case["call"] == "prefix":
            case["prefix"] = max(16, _log(rng, max(32, lo // 2), max(32, hi)))
            case["near"] = 0.0
            case["copy"] = min(case["copy"], 0.5)
    return case


# ----------------------------------------------------------------------------- inputs

_ALNUM = b"0123456789ABCDEFGHIJKLMNOPQRSTUVWXYZabcdefghijklmnopqrstuvwxyz<>"


def _fill(arena, nbytes, text, gen):
    """Random key bytes of the alphabet."""
    for a in range(0, nbytes, CHUNK):
        part = arena[a:min(nbytes, a + CHUNK)]
        if text == "printable":
            part.random_(0x20, 0x7F, generator=gen)
        else:
            chars = b"ACGT" if text == "acgt" else _ALNUM
            lut = torch.tensor(list(chars), dtype=torch.uint8, device=DEV)
            part.random_(0, len(chars), generator=gen)
            part.copy_(lut[part.int()])


def _lengths(n, lo, hi, gen):
    """Uniform over lo..hi in random order; the lengths as a whole are the same for every seed."""
    return lo + torch.randperm(n, device=DEV, generator=gen) * (hi - lo + 1) // n


def _offsets(lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=off[1:])
    return off


def _arena(nbytes):
    """Padded to a multiple of 16 bytes and 16 more, as every relation of this package."""
    arena = torch.empty((nbytes + 15) // 16 * 16 + 16, dtype=torch.uint8, device=DEV)
    arena[nbytes:] = 0
    return arena


def _copy_keys(dst, dst_at, src, src_at, lens):
    """dst[dst_at[i] : + lens[i]] = src[src_at[i] : + lens[i]] for every i."""
    ends = torch.cumsum(lens, 0)
    total = int(ends[-1]) if lens.numel() else 0
    cuts = torch.searchsorted(ends, torch.arange(0, total + CHUNK, CHUNK, device=DEV)).cpu().tolist()
    cuts = [min(c, lens.numel()) for c in cuts] + [lens.numel()]
    for a, b in zip(cuts, cuts[1:]):
        if b > a:
            part = lens[a:b]
            starts = torch.cumsum(part, 0) - part
            at = torch.arange(int(part.sum()), device=DEV)
            to = at + torch.repeat_interleave(dst_at[a:b] - starts, part)
            at += torch.repeat_interleave(src_at[a:b] - starts, part)
            dst[to] = src[at]


def _relations(shapes, text, copy, near, zipf, gen):
    """R and S of the joins `shapes` = [(m, n, lo, hi), ...] back to back, with row ranges."""
    lens_r, lens_s, rows, src, ranges, far = [], [], [], [], [], []
    r0 = s0 = 0
    for m, n, lo, hi in shapes:
        lr, ls = _lengths(m, lo, hi, gen), _lengths(n, lo, hi, gen)
        order = torch.randperm(n, device=DEV, generator=gen)
        k, k2 = int(copy * n), int(near * n)
        if zipf:
            w = torch.cumsum(torch.arange(1, m + 1, device=DEV, dtype=torch.float64) ** -zipf, 0)
            rank = torch.searchsorted(w, torch.rand(k + k2, device=DEV, dtype=torch.float64, generator=gen) * w[-1])
            partner = torch.randperm(m, device=DEV, generator=gen)[rank.clamp_(max=m - 1)]
        else:
            partner = torch.randint(0, m, (k + k2,), device=DEV, generator=gen)
        which = order[:k + k2]
        ls[which] = lr[partner]
        lens_r.append(lr)
        lens_s.append(ls)
        rows.append(which + s0)
        far.append(which[k:] + s0)
        src.append(partner + r0)
        ranges.append((r0, r0 + m, s0, s0 + n))
        r0, s0 = r0 + m, s0 + n
    lens_r, lens_s = torch.cat(lens_r), torch.cat(lens_s)
    off_r, off_s = _offsets(lens_r), _offsets(lens_s)
    a_r, a_s = _arena(int(off_r[-1])), _arena(int(off_s[-1]))
    _fill(a_r, int(off_r[-1]), text, gen)
    _fill(a_s, int(off_s[-1]), text, gen)
    rows, src, far = torch.cat(rows), torch.cat(src), torch.cat(far)
    _copy_keys(a_s, off_s[rows], a_r, off_r[src], lens_s[rows])
    if far.numel():                                # near-duplicates: one to six characters changed
        edits = torch.randint(1, 7, (far.numel(),), device=DEV, generator=gen)
        for j in range(6):
            some = far[edits > j]
            at = off_s[some] + (torch.rand(some.numel(), device=DEV, dtype=torch.float64, generator=gen)
                                * lens_s[some]).long()
            a_s[at] = torch.where(a_s[at] == 65, 67, 65).to(torch.uint8)
    return ag.DeviceRelation(a_r, off_r), ag.DeviceRelation(a_s, off_s), ranges


def _batch_shapes(case):
    """Sizes and key-length bands of a batch: a pure function of the case."""
    rng = random.Random("%d %d %d" % (case["joins"], case["median"], case["factor"]))
    shapes = []
    for j in range(case["joins"]):
        m = int(min(100_000, max(1000, rng.lognormvariate(math.log(case["median"]), 1.0))))
        shapes.append((m, case["factor"] * m) + BATCH_BANDS[j % 3])
    return shapes


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    st = {"case": case}
    op = case["op"]
    if op in ("sig", "gf8", "prefixes"):
        off = _offsets(_lengths(case["n"], case["lo"], case["hi"], gen))
        arena = _arena(int(off[-1]))
        _fill(arena, int(off[-1]), case["text"], gen)
        st["rel"] = ag.DeviceRelation(arena, off)
        if op != "prefixes":
            st["out"] = torch.empty(case["n"], dtype=torch.int64, device=DEV)
        return st
    if op == "batch":
        shapes = _batch_shapes(case)
        R, S, ranges = _relations(shapes, case["text"], case["copy"], 0.0, 0.0, gen)
        if case["gaps"]:                           # a request that takes every other join of the resident pool
            ranges = ranges[::2]
        caps = [max(64, se - sb) for (_, _, sb, se) in ranges]
        mr, ns = R.off.numel() - 1, S.off.numel() - 1
        R.ids = torch.arange(mr, dtype=torch.int32, device=DEV)
        S.ids = torch.arange(ns, dtype=torch.int32, device=DEV)
        st["descs"] = ag.make_descs(ranges, caps)
        st["ws"] = ag.alloc_ws(ag.join_batch_ws_bytes(st["descs"], mr, ns))
        st["batch"] = ag.join_batch_prepare(st["descs"], R, S, st["ws"])
        st["pairs"] = torch.empty(2 * ag.total_pair_cap(st["descs"]), dtype=torch.int32, device=DEV)
        st["counts"] = torch.zeros(len(ranges), dtype=torch.int64, device=DEV)
    else:
        m, n = case["m"], case["n"]
        R, S, _ = _relations([(m, n, case["lo"], case["hi"])], case["text"], case["copy"], case["near"],
                             case["zipf"], gen)
        st["pairs"] = torch.empty(2 * (n + m), dtype=torch.int32, device=DEV)
        st["count"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        if op == "probe":
            st["ws"] = ag.alloc_ws(ag.join_table_bytes(m))
            st["table"] = ag.join_build(R, st["ws"])
            st["sig"] = torch.empty(n, dtype=torch.int64, device=DEV)
        elif case["call"] == "into":
            st["ws"] = ag.alloc_ws(ag.join_ws_bytes(m, n))
        elif case["call"] == "prefix":
            st["ws"] = ag.alloc_ws(ag.join_prefix_ws_bytes(m, n))
        elif case["call"] == "partitioned":
            st["ws"] = ag.alloc_ws(ag.join_part_ws_bytes(m, n))
    st["R"], st["S"] = R, S
    rows = case["m"] if case.get("call") in ("semi_r", "anti_r") else S.n
    st["column"] = torch.empty(rows, dtype=torch.int32, device=DEV)
    return st


# ----------------------------------------------------------------------------- one pass

def _column(column, pairs):
    """The R row (or -1) of every S row, from the pairs (r, s)."""
    return column.fill_(-1).scatter_(0, pairs[:, 1].long(), pairs[:, 0])


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "sig":
        return ag.sig_compute(st["rel"], st["out"], n_components=case["ncomp"])
    if op == "gf8":
        return ag.sig_compute_gf8(st["rel"], st["out"])
    if op == "prefixes":
        return ag.sig_prefixes(st["rel"], case["block"])
    R, S, pairs = st["R"], st["S"], st["pairs"]
    if op == "batch":
        ag.join_batch_run(st["batch"], R, S, pairs, st["counts"])
        found = zip(st["descs"], st["counts"].cpu().tolist())
        both = torch.cat([pairs[2 * d.pair_offset: 2 * (d.pair_offset + c)] for d, c in found])
        return {"counts": st["counts"], "column": _column(st["column"], both.view(-1, 2))}
    call = case["call"]
    if op == "probe":
        if call == "inner":
            cnt = ag.join_probe(st["table"], S, pairs, st["count"], sigS_out=st["sig"])
        else:
            ag.sig_compute(S, st["sig"])
            cnt = ag.join_probe_mode(st["table"], S, st["sig"], pairs, st["count"], mode=call)
        got = pairs[:2 * cnt].view(-1, 2)
        if call in ("semi", "anti"):               # the selected S rows
            col = st["column"].fill_(0).index_fill_(0, got[:, 1].long(), 1)
        elif call in ("semi_r", "anti_r"):         # the selected R rows
            col = st["column"].fill_(0).index_fill_(0, got[:, 0].long(), 1)
        else:
            col = _column(st["column"], got)
        return {"count": cnt, "column": col, "sig": st["sig"]}
    if call == "join":
        got = ag.join(R, S)
        return {"count": got.shape[0], "column": _column(st["column"], got)}
    if call == "prefix":
        _, cnt = ag.join_prefix_into(R, S, case["prefix"], st["ws"], pairs, st["count"])
    elif call == "partitioned":
        _, cnt = ag.join_partitioned_into(R, S, st["ws"], pairs, st["count"])
    else:
        _, cnt = ag.join_into(R, S, st["ws"], pairs, st["count"])
    return {"count": cnt, "column": _column(st["column"], pairs[:2 * cnt].view(-1, 2))}


def work(case):
    """Bytes that a pass cannot do without: every key byte and offset read once, results written once."""
    op = case["op"]
    if op == "batch":
        shapes = _batch_shapes(case)[::2 if case["gaps"] else 1]
        total = sum((m + n) * (0.5 * (lo + hi) + 8) + n * (4 + 8 * case["copy"]) for m, n, lo, hi in shapes)
        return {"bytes": total, "flops": 0}
    mean = 0.5 * (case["lo"] + case["hi"])
    if op in ("sig", "gf8"):
        return {"bytes": case["n"] * (mean + 16), "flops": 0}
    if op == "prefixes":
        return {"bytes": case["n"] * (mean + 16 + 8 * (mean / case["block"] + 0.5)), "flops": 0}
    m, n = case["m"], case["n"]
    if op == "probe":                              # R's keys are read where a row has a partner
        return {"bytes": n * (mean + 8 + 8 + 12) + min(m, case["copy"] * n) * mean, "flops": 0}
    if case["call"] == "prefix":
        lo, hi, cap = case["lo"], case["hi"], case["prefix"]
        if cap < hi:
            mean = cap if cap <= lo else ((cap - lo) * 0.5 * (lo + cap) + (hi - cap) * cap) / (hi - lo)
    return {"bytes": (m + n) * (mean + 8) + n * (4 + 8 * case["copy"]), "flops": 0}


def exact(case, seed):
    """Every output is a whole number and has one right value: there is nothing to say in 64 bits."""
    return None
