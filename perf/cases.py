"""Performance cases of the RID recognizer: what a program that uses it calls, over the range it
calls it on.

Every case goes through the package's public entry points.  Texts are made on the GPU from the seed
alone (whole records or members of the RE's language, some with byte substitutions); results are
accept bits, chunk maps and entry sets, all whole numbers.
"""
import math
import random

import numpy as np
import torch

import paper_2412_14975_gb300 as rid

DEV = "cuda:0"

_TS = "[0-9]{4}-[0-9]{2}-[0-9]{2}T[0-9]{2}:[0-9]{2}:[0-9]{2}"
_ID = "[0-9]{1,9}"
_FLOAT = "[0-9]+\\.[0-9]{1,6}"
_WORD = "[a-z]{1,12}"
_IP = "[0-9]{1,3}\\.[0-9]{1,3}\\.[0-9]{1,3}\\.[0-9]{1,3}"
_FIELD = "(" + "|".join([_TS, _ID, _FLOAT, _WORD, _IP]) + ")"

# name: (RE, interface slots of the RI-DFA, states of the minimal DFA)
RES = {
    "pairs": ("([0-9]+,[a-z]+\n)*", 4, 4),                                # two-field lines
    "walk": ("((A|C)*G(T|A)+C)*", 4, 4),                                  # small alphabet, small automaton
    "records": ("(" + ",".join([_TS, _ID, _FLOAT, _WORD, _IP]) + "\\n)*", 68, 68),   # record lines
    "anyfield": ("(" + _FIELD + "(," + _FIELD + ")*\\n)*", 54, 53),       # any field in any column
    "codon": ("(([ACGT]{3})*ATG([ACGT]{3}){2,4}(TAA|TAG|TGA))*[ACGT]*", 24, 1),      # runs that stay apart
}
for _k in range(3, 10):
    RES["regexp%d" % _k] = ("(a|b)*a(a|b){%d}" % _k, _k + 2, 2 ** (_k + 1))

# one record of each generated text as segments: (kind, fixed byte or None, shortest, longest);
# kinds: digit, letter, fixed, and three two- or four-letter alphabets
_DIGIT, _LETTER, _FIXED, _AC, _TA, _ACGT, _AB = range(7)
_KINDS = {_DIGIT: b"0123456789", _LETTER: b"abcdefghijklmnopqrstuvwxyz", _AC: b"AC", _TA: b"TA",
          _ACGT: b"ACGT", _AB: b"ab"}


def _fix(c):
    return (_FIXED, ord(c), 1, 1)


def _d(lo, hi):
    return (_DIGIT, 0, lo, hi)


_SEG_TS = [_d(4, 4), _fix("-"), _d(2, 2), _fix("-"), _d(2, 2), _fix("T"), _d(2, 2), _fix(":"), _d(2, 2), _fix(":"), _d(2, 2)]
_SEG_IP = [_d(1, 3), _fix("."), _d(1, 3), _fix("."), _d(1, 3), _fix("."), _d(1, 3)]
_RECORDS = {
    "pairs": [_d(1, 6), _fix(","), (_LETTER, 0, 1, 8), _fix("\n")],
    # (A|C)* G (T|A)+ C with the run lengths of a uniform walk on the minimal DFA (see _lengths)
    "walk": [(_AC, 0, 0, -1), _fix("G"), (_TA, 0, 1, -1), _fix("C")],
    "records": _SEG_TS + [_fix(","), _d(1, 9), _fix(","), _d(1, 9), _fix("."), _d(1, 6), _fix(","),
                          (_LETTER, 0, 1, 12), _fix(",")] + _SEG_IP + [_fix("\n")],
}
_RECORDS["anyfield"] = _RECORDS["records"]


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _letters(kind, n, g):
    lut = torch.tensor(list(_KINDS[kind]), dtype=torch.uint8, device=DEV)
    return lut[torch.randint(0, lut.numel(), (n,), generator=g, device=DEV)]


def _lengths(lo, hi, n, g):
    if hi < 0:       # each further letter with probability 2/3 (from 0) or 2/3 after the first
        p = 2.0 / 3.0
        u = torch.rand(n, generator=g, device=DEV).clamp_(min=1e-12)
        return lo + (torch.log(u) / math.log(p)).floor().to(torch.int64).clamp_(max=200)
    return torch.randint(lo, hi + 1, (n,), generator=g, device=DEV)


def _record_text(segs, n, g, block=1 << 20):
    """Whole records until at least n bytes."""
    kind = torch.tensor([k for k, _, _, _ in segs], dtype=torch.uint8, device=DEV)
    fixed = torch.tensor([f for _, f, _, _ in segs], dtype=torch.uint8, device=DEV)
    mean = sum((3.0 if hi < 0 else (lo + hi) / 2.0) for _, _, lo, hi in segs)
    parts, total = [], 0
    while total < n:
        nrec = int(min(block, max(4, (n - total) / mean * 1.02 + 64)))
        lens = torch.stack([_lengths(lo, hi, nrec, g) for _, _, lo, hi in segs], dim=1)
        seg = torch.repeat_interleave(torch.arange(len(segs), device=DEV, dtype=torch.uint8).repeat(nrec), lens.reshape(-1))
        out = fixed[seg.to(torch.int32)]
        kd = kind[seg.to(torch.int32)]
        for k in {s[0] for s in segs} - {_FIXED}:
            out = torch.where(kd == k, _letters(k, out.numel(), g), out)
        if total + out.numel() > n:
            ends = torch.cumsum(lens.sum(1), 0)
            out = out[:int(ends[int(torch.searchsorted(ends, n - total))])]
        parts.append(out)
        total += out.numel()
    return torch.cat(parts)


def _text(name, n, seed, subs, offset):
    """A member of RES[name]'s language of at least n bytes (exactly n where any length is one),
    `subs` bytes of it substituted, starting `offset` bytes past a 16-byte boundary."""
    g = _gen(seed)
    if name in _RECORDS:
        x = _record_text(_RECORDS[name], n, g)
    elif name == "codon":
        x = _letters(_ACGT, n, g)
    else:
        x = _letters(_AB, n, g)
        k = int(name[6:])
        if n > k:
            x[n - k - 1] = ord("a")          # the (k+1)-th byte from the end decides
    if subs:
        at = torch.randint(0, x.numel(), (subs,), generator=g, device=DEV)
        x[at] = x[torch.randint(0, x.numel(), (subs,), generator=g, device=DEV)]
    if offset:
        buf = torch.empty(x.numel() + 16, dtype=torch.uint8, device=DEV)
        buf[offset:offset + x.numel()] = x
        x = buf[offset:offset + x.numel()]
    return x


# ------------------------------------------------------------- many texts against many REs
# Random (R)* REs, as a service that holds its users' patterns meets them: alphabets of 4 to 64
# symbols, depth 6, union, concatenation, star and bounded repeat, RI-DFAs of 10 to 5,000 states.
# (The seeds whose RE falls outside those limits are left out; the others are the first ones.)
_RE_SEEDS = (2, 3, 4, 5, 6, 8, 9, 11, 14, 16, 17, 20, 21, 23, 24, 27, 30, 32, 34, 35, 37, 39, 41, 43, 45, 48, 49, 50, 53)


def _leaf(r, alphabet):
    if len(alphabet) > 1 and r.random() < 0.3:
        return ("sym", sorted(r.sample(alphabet, r.randint(2, min(len(alphabet), 4)))))
    return ("sym", [r.choice(alphabet)])


def _tree(r, alphabet, depth):
    if depth <= 0 or r.random() < 0.2:
        return _leaf(r, alphabet)
    x = r.random()
    if x < 0.6:
        return ("cat" if x < 0.35 else "alt", [_tree(r, alphabet, depth - 1) for _ in range(r.randint(2, 3))])
    if x < 0.85:
        return ("star", _tree(r, alphabet, depth - 1))
    lo = r.randint(0, 3)
    return ("rep", _tree(r, alphabet, depth - 1), lo, max(1, lo + r.randint(0, 5)))


def _render(t):
    if t[0] == "sym":
        s = "".join("\\x%02x" % b for b in t[1])
        return s if len(t[1]) == 1 else "[" + s + "]"
    if t[0] == "cat":
        return "".join("(" + _render(i) + ")" for i in t[1])
    if t[0] == "alt":
        return "|".join("(" + _render(i) + ")" for i in t[1])
    return "(" + _render(t[1]) + ")" + ("*" if t[0] == "star" else "{%d,%d}" % (t[2], t[3]))


def _member(t, r, out):
    if t[0] == "sym":
        out.append(r.choice(t[1]))
    elif t[0] == "cat":
        for i in t[1]:
            _member(i, r, out)
    elif t[0] == "alt":
        _member(r.choice(t[1]), r, out)
    elif t[0] == "star":
        while len(out) < 64 and r.random() < 0.6:
            _member(t[1], r, out)
    else:
        for _ in range(r.randint(t[2], t[3])):
            _member(t[1], r, out)


def _random_re(seed):
    r = random.Random(seed)
    alphabet = list(range(0x21, 0x21 + r.randint(4, 64)))
    t = _tree(r, alphabet, 6)
    return "(" + _render(t) + ")*", t


def _collection(count):
    """The REs of a many-text workload: records, walk, codon and random ones."""
    return [("records", None), ("walk", None), ("codon", None)] + [("random", s) for s in _RE_SEEDS[:count - 3]]


def _source(kind, re_seed):
    return RES[kind][0] if kind != "random" else _random_re(re_seed)[0]


def _long_text(kind, re_seed, n, seed):
    """A text of at least n bytes of the RE's language and the ascending ends of its members (text
    boundaries fall on them)."""
    g = _gen(seed)
    if kind == "codon":
        return _letters(_ACGT, n, g), None
    if kind != "random":
        x = _record_text(_RECORDS[kind], n, g)
        last = 10 if kind == "records" else ord("C")
        ends = torch.nonzero(x == last).flatten() + 1
        if kind == "walk":                    # a C right after a T always ends a member
            ends = ends[x[(ends - 2).clamp_(min=0)] == ord("T")]
        return x, ends
    r = random.Random(re_seed * 7919 + 1)
    tree = _random_re(re_seed)[1]
    pool = []
    for _ in range(400):
        m = []
        _member(tree, r, m)
        if m:
            pool.append(m)
    lens = torch.tensor([len(m) for m in pool], device=DEV)
    offs = torch.cumsum(lens, 0) - lens
    data = torch.tensor([b for m in pool for b in m], dtype=torch.uint8, device=DEV)
    idx = torch.randint(0, len(pool), (int(n / float(lens.float().mean()) * 1.1) + 64,), generator=g, device=DEV)
    ls = lens[idx]
    ends = torch.cumsum(ls, 0)
    at = torch.repeat_interleave(offs[idx] - (ends - ls), ls) + torch.arange(int(ends[-1]), device=DEV)
    return data[at], ends


def _many_texts(res, count, median, largest, seed):
    """count texts of lognormal length (sigma 1), text j of RE j mod len(res), every other one with
    one byte substituted: (device tensor, RE index) per text, in order."""
    h = np.random.Generator(np.random.PCG64(seed))
    want = np.clip(np.exp(h.normal(math.log(median), 1.0, count)), 1 << 10, largest).astype(np.int64)
    texts = [None] * count
    for r, (kind, re_seed) in enumerate(res):
        mine = list(range(r, count, len(res)))
        if not mine:
            continue
        cuts = np.cumsum(want[mine])
        x, ends = _long_text(kind, re_seed, int(cuts[-1]), seed * 131 + r)
        if ends is not None:
            at = torch.searchsorted(ends, torch.from_numpy(cuts).to(DEV)).clamp_(max=ends.numel() - 1)
            cuts = ends[at].cpu().numpy()
        lo = 0
        for j, hi in zip(mine, cuts):
            texts[j] = x[lo:int(hi)]
            lo = int(hi)
    size = [t.numel() for t in texts]
    offs = np.zeros(count + 1, dtype=np.int64)
    np.cumsum([(s + 15) & ~15 for s in size], out=offs[1:])
    buf = torch.zeros(int(offs[-1]) + 16, dtype=torch.uint8, device=DEV)
    for j, t in enumerate(texts):
        buf[int(offs[j]):int(offs[j]) + size[j]] = t
    hit = [j for j in range(1, count, 2) if size[j] > 1]
    to = torch.tensor([int(offs[j]) + int(h.integers(size[j])) for j in hit], device=DEV)
    frm = torch.tensor([int(offs[j]) + int(h.integers(size[j])) for j in hit], device=DEV)
    buf[to] = buf[frm]
    return [(buf[int(offs[j]):int(offs[j]) + size[j]], j % len(res)) for j in range(count)]


# ------------------------------------------------------------------------------- the cases
KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30


def _one(name, re, n, chunks, call="recognize", dfa=False, subs=0, offset=0):
    return {"name": name, "kind": "text", "re": re, "bytes": n, "chunks": chunks, "call": call, "dfa": dfa,
            "subs": subs, "offset": offset}


def listed():
    return [
        # a short message in a few chunks: the smallest call, all latency
        _one("pairs_4k", "pairs", 4093, 4),
        # the plain configuration: 1 MiB in 64 chunks, a small automaton
        _one("walk_1m", "walk", MIB, 64),
        # a log file of ordinary size
        _one("records_64m", "records", 64 * MIB, 16384),
        # a large log file, more than L2 holds many times over: the headline workload's shape
        _one("records_4g", "records", 4 * GIB, 155648, call="async"),
        # the same language family with a larger automaton, an odd size, a chunk count that is not
        # a multiple of the lanes
        _one("anyfield_1g", "anyfield", GIB + 4099, 131072, call="async", subs=1),
        # the all-states DFA, the method's comparator
        _one("records_dfa_512m", "records", 512 * MIB, 131072, dfa=True),
        # genome-like text in many and in few chunks: runs that never merge
        _one("codon_1g_64k", "codon", GIB, 65536, call="async"),
        _one("codon_1g_4k", "codon", GIB, 4096, subs=2),
        # the paper's regexp family, where the interface is far smaller than the DFA
        _one("regexp7_1g", "regexp7", GIB, 131072, call="async"),
        # where was my text rejected: recognition with maps, then the join as a scan; the text is a
        # slice of a larger buffer (not 16-byte aligned)
        _one("records_scan_256m", "records", 256 * MIB, 65537, call="scan", subs=1, offset=5),
        # many texts of uneven length against many REs: one graph launch
        {"name": "batch_2000x16", "kind": "batch", "texts": 2000, "res": 16, "median": 256 * KIB, "chunk_len": 0},
        # a burst of requests at a server that holds many REs
        {"name": "served_64", "kind": "served", "texts": 64, "res": 32, "median": 64 * KIB},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    x = rng.random()
    if x < 0.12:
        return {"kind": "batch", "texts": _log(rng, 50, 2000), "res": rng.choice([3, 8, 16]),
                "median": _log(rng, 16 * KIB, 256 * KIB), "chunk_len": rng.choice([0, 0, 8192])}
    if x < 0.2:
        return {"kind": "served", "texts": _log(rng, 1, 128), "res": rng.choice([8, 32]), "median": _log(rng, 8 * KIB, 128 * KIB)}
    re = rng.choice(["pairs", "walk", "records", "records", "anyfield", "codon", "codon"] + ["regexp%d" % rng.randint(3, 9)])
    n = _log(rng, 4 * KIB, GIB) | 1
    chunks = max(4, min(_log(rng, 4, 1 << 20), n // 64))
    if re == "codon":
        chunks = max(chunks, n >> 18)         # configured: 2^12 to 2^20 chunks of 1 GiB
    dfa = re not in ("codon", "regexp8", "regexp9") and rng.random() < 0.15
    call = "recognize" if dfa else rng.choice(["recognize", "recognize", "async", "async", "scan"])
    c = _one("", re, n, chunks, call=call, dfa=dfa, subs=rng.choice([0, 0, 1, 8]), offset=rng.choice([0, 0, 0, rng.randint(1, 15)]))
    del c["name"]
    return c


def prepare(case, seed):
    if case["kind"] == "text":
        src, k, q = RES[case["re"]]
        prog = rid.ridfa_compile(src)
        x = _text(case["re"], case["bytes"], seed, case["subs"], case["offset"])
        width = q if case["dfa"] else k
        st = {"case": case, "prog": prog, "text": x, "n": x.numel(), "c": case["chunks"],
              "maps": torch.empty((case["chunks"], width), dtype=torch.int16, device=DEV),
              "accept": torch.zeros(1, dtype=torch.uint8, device=DEV)}
        if case["call"] == "scan":
            st["entry"] = torch.empty((case["chunks"], (k + 31) // 32), dtype=torch.int32, device=DEV)
        return st
    res = _collection(case["res"])
    progs = [rid.ridfa_compile(_source(*r), build_dfa=False) for r in res]
    if case["kind"] == "batch":
        texts = _many_texts(res, case["texts"], case["median"], 64 * MIB, seed)
        accept = torch.zeros(len(texts), dtype=torch.uint8, device=DEV)
        items = [(t, t.numel(), r, 0) for t, r in texts]
        return {"case": case, "texts": texts, "accept": accept,
                "batch": rid.ridfa_batch_create(progs, items, accept, chunk_len=case["chunk_len"])}
    texts = _many_texts(res, case["texts"], case["median"], 16 * MIB, seed)
    srv = rid.Server(arena_bytes=256 * MIB)
    slots = [srv.add_program(p) for p in progs]
    return {"case": case, "server": srv, "texts": [(slots[r], t.cpu().numpy()) for t, r in texts]}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        rid.ridfa_batch_run(state["batch"])
        return state["accept"]
    if case["kind"] == "served":
        srv = state["server"]
        ids = {srv.submit(slot, x): i for i, (slot, x) in enumerate(state["texts"])}
        accept, status, left = np.zeros(len(ids), dtype=np.uint8), np.zeros(len(ids), dtype=np.int32), len(ids)
        while left:
            for req, err, acc, _ in srv.poll(wait_us=1000):
                accept[ids[req]], status[ids[req]] = acc, err
                left -= 1
        return {"accept": accept, "status": status}
    prog, x, n, c, maps = state["prog"], state["text"], state["n"], state["c"], state["maps"]
    if case["call"] == "async":
        rid.ridfa_recognize_async(prog, x, n, c, state["accept"], d_chunk_maps=maps)
        return {"accept": state["accept"], "maps": maps}
    call = rid.ridfa_recognize_dfa if case["dfa"] else rid.ridfa_recognize
    out = {"accept": call(prog, x, n, c, d_chunk_maps=maps), "maps": maps}
    if case["call"] == "scan":
        out["first_reject"] = rid.ridfa_join_scan(prog, maps, c, d_entry=state["entry"])
        out["entry"] = state["entry"]
    return out


def work(case):
    if case["kind"] != "text":
        n = case["texts"] * case["median"] * math.exp(0.5)      # the lognormal's mean
        return {"bytes": n + case["texts"], "flops": 0}
    _, k, q = RES[case["re"]]
    b = case["bytes"] + 2 * case["chunks"] * (q if case["dfa"] else k)
    if case["call"] == "scan":      # the scan reads the maps and writes the entry sets
        b += case["chunks"] * (2 * k + 4 * ((k + 31) // 32))
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Accept bits, states and sets are whole numbers, equal or wrong: nothing is computed in floating point."""
    return None
