"""Measured cases: the calls a program makes to this library, over its range of sizes.

A case names an operation, a regular expression and sizes.  Texts are drawn on
the device from the distributions of the repository's workloads: web-server
log lines, DNA with planted reading frames, uniform a/b, and texts of random
regular expressions built from whole iterations of their outer star.
"""
import math
import random

import numpy as np
import torch

from paper_2503_06763_gb300 import Batch, Regex, ReError
from paper_2503_06763_gb300.native import slpf_dfa_decode, slpf_dfa_encode

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30

AB_RE = "(a|b|ab)*"
DNA_RE = "([ACGT]|ATG([ACGT][ACGT][ACGT])*(TAA|TAG|TGA))*"
DNA_STOP_GROUP = 13                     # the node (TAA|TAG|TGA) of DNA_RE

_MONTHS = "Jan Feb Mar Apr May Jun Jul Aug Sep Oct Nov Dec".split()
_METHODS = "GET POST PUT DELETE HEAD".split()
_OCTET, _D2 = "[0-9][0-9]?[0-9]?", "[0-9][0-9]"
LOG_GOOD = (
    f"{_OCTET}\\.{_OCTET}\\.{_OCTET}\\.{_OCTET} - - \\["
    f"{_D2}/({'|'.join(_MONTHS)})/[0-9][0-9][0-9][0-9]:{_D2}:{_D2}:{_D2} [+\\-][0-9][0-9][0-9][0-9]\\] "
    f"\"({'|'.join(_METHODS)}) /[a-zA-Z0-9_./\\-]* HTTP/1\\.[01]\" [1-5][0-9][0-9] [0-9]+"
)
LOG_RE = f"(({LOG_GOOD}|[^\\n]*)\\n)*"


# ----------------------------------------------------------------------------- texts
def _log_lines(seed, high, count=4096):
    """count log lines: 2 % malformed, a share ``high`` with a word of UTF-8 text."""
    r = random.Random(seed)
    letters = "abcdefghijklmnopqrstuvwxyz0123456789_"
    vocab = ["".join(r.choices(letters, k=r.randint(3, 11))) for _ in range(4000)]
    weights = [1.0 / (j + 1) for j in range(len(vocab))]
    toks = iter(r.choices(vocab, weights, k=3 * count))
    out = []
    for _ in range(count):
        u = r.random()
        method = "GET" if u < 0.80 else "POST" if u < 0.95 else r.choice(_METHODS[2:])
        path = "/" + "/".join(next(toks) for _ in range(r.randint(1, 3)))
        status = 200 if r.random() < 0.9 else r.choice((301, 302, 304, 400, 403, 404, 500, 503))
        line = ("%d.%d.%d.%d - - [%02d/%s/%d:%02d:%02d:%02d %s%04d] \"%s %s HTTP/1.%d\" %d %d" % (
            r.randrange(256), r.randrange(256), r.randrange(256), r.randrange(256), r.randint(1, 28),
            r.choice(_MONTHS), r.randint(1995, 2025), r.randrange(24), r.randrange(60), r.randrange(60),
            r.choice("+-"), r.randrange(1300), method, path, r.randrange(2), status,
            r.randrange(1, 10 ** r.randint(1, 7))))
        if r.random() < 0.02:
            j = r.randrange(1, len(line))
            line = r.choice((line[:j], line[:j] + chr(r.randint(32, 126)) + line[j + 1:], line.replace('"', "", 1)))
        if r.random() < high:
            line += " café naïve 你好"
        out.append(line.encode("utf-8") + b"\n")
    return out


class _Node:
    """A random regular expression as a tree: its pattern and random texts of it."""

    def __init__(self, r, budget, depth, stars, alphabet):
        u = r.random()
        self.kids = []
        if budget <= 1 or depth > 12:
            self.kind, self.sym = "sym", r.choice(alphabet)
            return
        self.kind = "alt" if u < 0.3 else "cat" if u < 0.8 or stars >= 3 else "star"
        if self.kind == "star":
            for _ in range(20):
                body = _Node(r, budget - 1, depth + 1, stars + 1, alphabet)
                if not body.nullable():
                    self.kids = [body]
                    return
            self.kind = "cat"
        cuts = [r.expovariate(1.0) for _ in range(r.randint(2, 3))]
        self.kids = [_Node(r, max(1, int(budget * c / sum(cuts))), depth + 1, stars, alphabet) for c in cuts]

    def nullable(self):
        if self.kind in ("sym", "star"):
            return self.kind == "star"
        return (all if self.kind == "cat" else any)(k.nullable() for k in self.kids)

    def positions(self):
        return 1 if self.kind == "sym" else sum(k.positions() for k in self.kids)

    def pattern(self):
        if self.kind == "sym":
            return self.sym
        if self.kind == "star":
            return "(" + self.kids[0].pattern() + ")*"
        return "(" + ("|" if self.kind == "alt" else "").join(k.pattern() for k in self.kids) + ")"

    def emit(self, r, out):
        if self.kind == "sym":
            out.append(self.sym)
        elif self.kind == "cat":
            for k in self.kids:
                k.emit(r, out)
        elif self.kind == "alt":
            r.choice(self.kids).emit(r, out)
        else:
            while r.random() < 0.5 and len(out) < 1 << 16:
                self.kids[0].emit(r, out)


def _regen(seed, lo, hi):
    """The body of a random RE (body)* of lo..hi positions over 8 to 48 letters,
    one whose tables the library's limits admit."""
    r = random.Random(seed)
    pool = "abcdefghijklmnopqrstuvwxyzABCDEFGHIJKLMNOPQRSTUVWXYZ0123456789!#%&,:;<=>@_~"
    while True:
        alphabet = r.sample(pool, r.randint(8, 48))
        body = _Node(r, r.randint(lo, hi), 0, 1, alphabet)
        if body.nullable() or not lo <= body.positions() <= hi:
            continue
        try:
            Regex("(" + body.pattern() + ")*", host_only=True).close()
        except ReError:
            continue
        return body


def _pieces_of(body, seed, count=1024):
    r = random.Random(seed)
    out = []
    for _ in range(count):
        part = []
        body.emit(r, part)
        out.append("".join(part).encode("latin-1"))
    return sorted(out, key=len)


class _Pool:
    """Pieces (in order of length) on the device; text(n): at most n bytes of
    whole pieces.  The sequence of lengths comes from ``layout`` alone, which
    piece of a length stands there from ``seed``, so texts of every seed are
    equally long."""

    def __init__(self, pieces, layout, seed):
        lens = np.array([len(p) for p in pieces], dtype=np.int64)
        self.mean = float(lens.mean())
        first = np.searchsorted(lens, lens, side="left")
        same = np.searchsorted(lens, lens, side="right") - first
        self.lens, self.first, self.same = (torch.from_numpy(v).cuda() for v in (lens, first, same))
        self.starts = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)[:-1]])).cuda()
        self.data = torch.frombuffer(bytearray(b"".join(pieces)), dtype=torch.uint8).cuda()
        self.gens = [torch.Generator(device="cuda") for _ in range(2)]
        self.gens[0].manual_seed(layout)
        self.gens[1].manual_seed(seed)

    def _part(self, n):
        count = int(n / self.mean * 1.2) + 64
        while True:
            idx = torch.randint(0, self.lens.numel(), (count,), generator=self.gens[0], device="cuda")
            ends = self.lens[idx].cumsum(0)
            if int(ends[-1]) >= n:
                break
            count *= 2
        keep = int(torch.searchsorted(ends, n, right=True))
        if not keep:
            return torch.empty(0, dtype=torch.uint8, device="cuda")
        idx, ends = idx[:keep], ends[:keep]
        u = torch.rand(keep, generator=self.gens[1], device="cuda", dtype=torch.float64)
        idx = self.first[idx] + (u * self.same[idx]).long()
        ln = self.lens[idx]
        src = torch.repeat_interleave(self.starts[idx] - (ends - ln), ln)
        src += torch.arange(src.numel(), device="cuda")
        return self.data[src]

    def text(self, n):
        step, parts, left = 64 * MIB, [], n
        while left > 0:
            part = self._part(min(step, left))
            parts.append(part)
            if left <= step or not part.numel():
                break
            left -= part.numel()
        return torch.cat(parts)


def _log_text(n, seed, high):
    """n bytes of log lines; the last line is cut short (a file still being written)."""
    lines = sorted(_log_lines(seed, high), key=len)
    x = _Pool(lines, seed, seed).text(n + len(lines[-1]))[:n].clone()
    x[n - 1] = 10
    return x


def _dna_text(n, seed):
    """Uniform ACGT with reading frames (ATG, codons, a stop codon) about every 10 kB."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    acgt = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device="cuda")
    x = acgt[torch.randint(0, 4, (n,), generator=g, device="cuda", dtype=torch.uint8).int()]
    rng = np.random.Generator(np.random.PCG64(seed))
    count = n // 10_000 + 1
    codons = np.minimum(30 + rng.geometric(0.01, count), 900)
    starts = np.cumsum(rng.exponential(10_000, count).astype(np.int64) + 1 + 3 * np.concatenate([[0], codons[:-1]]))
    fits = starts + 3 * codons <= n
    codons, starts = torch.from_numpy(codons[fits]).cuda(), torch.from_numpy(starts[fits]).cuda()
    if codons.numel():
        every = [bytes((a, b, c)) for a in b"ACGT" for b in b"ACGT" for c in b"ACGT"]
        stops = [b"TAA", b"TAG", b"TGA"]
        table = torch.tensor([list(c) for c in [c for c in every if c not in stops] + stops + [b"ATG"]],
                             dtype=torch.uint8, device="cuda")
        ends = codons.cumsum(0)
        pick = torch.randint(0, 61, (int(ends[-1]),), generator=g, device="cuda")
        pick[ends - 1] = torch.randint(61, 64, (ends.numel(),), generator=g, device="cuda")
        pick[ends - codons] = 64
        first = torch.repeat_interleave(starts - 3 * (ends - codons), codons)
        at = first + 3 * torch.arange(pick.numel(), device="cuda")
        x[(at[:, None] + torch.arange(3, device="cuda")).reshape(-1)] = table[pick].reshape(-1)
    return x


def _pattern(case):
    re = case["re"]
    if re == "ab":
        return AB_RE
    if re == "dna":
        return DNA_RE
    if re == "log":
        return LOG_RE
    if re == "ek":                                   # the paper's family e(k): 2^(k+1) + 1 forward states
        return "(a|b)*a" + "(a|b)" * case["k"]
    return _pattern_of(_regen(case["re_seed"], 10, 200))


def _text(case, n, seed):
    re = case["re"]
    if re in ("ab", "ek"):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        x = torch.randint(97, 99, (n,), generator=g, device="cuda", dtype=torch.uint8)
        if re == "ek":
            x[n - 1 - case["k"]] = 97                # accepted: an a that many letters before the last
    elif re == "dna":
        x = _dna_text(n, seed)
    elif re == "log":
        x = _log_text(n, seed, case.get("high", 0.0))
    else:
        x = _Pool(_pieces_of(_regen(case["re_seed"], 10, 200), case["re_seed"]), n, seed).text(n)
    return x


# ----------------------------------------------------------------------------- cases
def listed():
    return [
        # a served request at the small end (a few dozen log lines): launches and latency
        {"name": "parse-log-4k", "op": "parse", "re": "log", "n": 4 * KIB + 37, "high": 0.0, "tune": False},
        # the ambiguous running example at 1 MiB, the latency benchmark
        {"name": "parse-ab-1m", "op": "parse", "re": "ab", "n": MIB, "tune": False},
        # a day's log file (11 MB), some lines with UTF-8 text: the default call
        {"name": "parse-log-11m", "op": "parse", "re": "log", "n": 11_182 * KIB + 11, "high": 0.02, "tune": False},
        # an RE of the e(k) family, whose forward automaton is too large for byte state ids
        {"name": "parse-ek9-16m", "op": "parse", "re": "ek", "k": 9, "n": 16 * MIB + 5, "tune": False},
        # a genome-sized text: the DNA workload
        {"name": "parse-dna-256m", "op": "parse", "re": "dna", "n": 256 * MIB, "tune": False},
        # the largest single text, parsed by a program that tunes once and keeps its buffers
        {"name": "parse-log-1g", "op": "parse", "re": "log", "n": GIB, "high": 0.0, "tune": True},
        # validation only: twelve uploaded logs, some cut off in mid line
        {"name": "recognize-log-24m", "op": "recognize", "re": "log", "n": 24 * MIB - 77, "high": 0.0},
        # a served batch: lognormal request lengths under 16 resident REs, planned and run on arrival
        {"name": "serve-48", "op": "serve", "re": "regen", "count": 48, "res": 16, "median": 64 * KIB, "re_seed": 11},
        # a planned batch run again over its bound buffers: lengths 1 KiB to 4 MiB under 8 REs
        {"name": "batch-768", "op": "batch", "re": "regen", "count": 768, "res": 8, "hi": 4 * MIB, "re_seed": 40},
        # every stop codon group of a DNA text from its parsed columns
        {"name": "matches-dna-64m", "op": "matches", "re": "dna", "n": 64 * MIB + 3},
        # a stored log's columns rebuilt on the device, and a log's columns stored
        {"name": "unarchive-log-48m", "op": "unarchive", "re": "log", "n": 48 * MIB, "high": 0.0, "interval": 4096},
        {"name": "archive-log-3m", "op": "archive", "re": "log", "n": 3 * MIB, "high": 0.0, "interval": 4096},
    ]


def _size(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    op = rng.choices(("parse", "recognize", "serve", "batch", "matches", "unarchive", "archive"),
                     (8, 2, 2, 2, 1, 1, 1))[0]
    if op == "serve":
        return {"op": op, "re": "regen", "count": _size(rng, 2, 96), "res": rng.randint(1, 16),
                "median": _size(rng, 8 * KIB, 128 * KIB), "re_seed": rng.randrange(1000)}
    if op == "batch":
        return {"op": op, "re": "regen", "count": _size(rng, 32, 768), "res": rng.randint(1, 8),
                "hi": _size(rng, 64 * KIB, 4 * MIB), "re_seed": rng.randrange(1000)}
    if op == "matches":
        return {"op": op, "re": "dna", "n": _size(rng, 16 * KIB, 64 * MIB)}
    if op in ("unarchive", "archive"):
        return {"op": op, "re": rng.choice(("log", "dna")), "n": _size(rng, 4 * KIB, (48 if op == "unarchive" else 3) * MIB),
                "high": 0.0, "interval": rng.choice((512, 1000, 4096))}
    re = rng.choice(("log", "log", "dna", "ab", "ek", "regen"))
    case = {"op": op, "re": re, "high": 0.0}
    top = {"log": GIB, "dna": 256 * MIB, "ab": 256 * MIB, "ek": 16 * MIB, "regen": 128 * MIB}[re]
    case["n"] = _size(rng, 2 * KIB, top if op == "parse" else min(top, 64 * MIB))
    case["tune"] = op == "parse" and case["n"] >= 64 * MIB and rng.random() < 0.5
    if re == "log":
        case["high"] = rng.choice((0.0, 0.02, 0.3))
    elif re == "ek":
        case["k"] = rng.randint(3, 11)
    elif re == "regen":
        case["re_seed"] = rng.randrange(1000)
    return case


def _bodies(case):
    return [_regen(1000 + 64 * case["re_seed"] + j, 10, 200) for j in range(case["res"])]


def _pattern_of(body):
    return "(" + body.pattern() + ")*"


def _lengths(case):
    rng = np.random.Generator(np.random.PCG64(case["re_seed"]))
    if case["op"] == "serve":
        lens = np.minimum(np.exp(rng.normal(math.log(case["median"]), 1.5, case["count"])), 4 * MIB)
    else:
        lens = np.exp(rng.uniform(math.log(KIB), math.log(case["hi"]), case["count"]))
    return lens.astype(np.int64), rng.integers(0, case["res"], case["count"])


def _prepare_batch(case, seed):
    """Texts under the case's REs, and one output arena that holds every text's columns."""
    bodies = _bodies(case)
    res = [Regex(_pattern_of(b)) for b in bodies]
    pools = [_Pool(_pieces_of(b, case["re_seed"] + j), case["re_seed"], seed + j) for j, b in enumerate(bodies)]
    lens, which = _lengths(case)
    texts = [pools[w].text(int(n)) for n, w in zip(lens, which)]
    rxs = [res[w] for w in which]
    sizes = [(rx.layout(t.numel())[1], rx.layout(t.numel())[2]) for rx, t in zip(rxs, texts)]
    offs = np.concatenate([[0], np.cumsum([(b + 255) // 256 * 256 for _, b in sizes])])
    arena = torch.zeros(int(offs[-1]), dtype=torch.uint8, device="cuda")
    dts = {1: torch.uint8, 2: torch.int16, 4: torch.int32, 8: torch.int64}
    outs = [arena[int(o):int(o) + b].view(dts[cb]) for o, (cb, b) in zip(offs, sizes)]
    status = torch.empty(len(texts), dtype=torch.int32, device="cuda")
    return {"op": case["op"], "texts": texts, "rxs": rxs, "arena": arena, "outs": outs, "status": status}


def prepare(case, seed):
    op = case["op"]
    if op in ("serve", "batch"):
        state = _prepare_batch(case, seed)
        if op == "batch":                               # planned and bound once
            state["batch"] = Batch(state["rxs"], [t.numel() for t in state["texts"]])
            state["batch"].parse(state["texts"], outs=state["outs"], status=state["status"])
        torch.cuda.synchronize()
        return state
    rx = Regex(_pattern(case))
    if op == "recognize":
        cut = random.Random(seed)
        texts = []
        for j in range(12):
            x = _text(case, case["n"], seed + 1000 * j)
            if cut.random() < 0.4:
                x[-1] = 1                               # no alternative ends there: rejected
            texts.append(x)
        torch.cuda.synchronize()
        return {"op": op, "rx": rx, "texts": texts}
    text = _text(case, case["n"], seed)
    n = text.numel()
    state = {"op": op, "rx": rx, "text": text, "n": n}
    if op == "parse" and n >= 64 * MIB:                  # a program of long texts keeps its buffers
        if case.get("tune"):
            rx.autotune(text)
        state["out"], state["status"], _ = rx.parse(text)
        state["workspace"] = torch.empty(rx.workspace_size(n), dtype=torch.uint8, device="cuda")
    elif op in ("matches", "archive", "unarchive"):
        state["cols"], state["status"], state["kind"] = rx.parse(text)
        if op == "matches":                             # room for the spans wanted; the total is reported too
            spans = n * 3 / 64
            state["cap"] = int(0.98 * spans - 8 * math.sqrt(spans))
        else:
            state["interval"] = case["interval"]
            state["host_cols"] = state["cols"].cpu().numpy()
            state["host_text"] = text.cpu().numpy()
            if op == "unarchive":
                state["archive"] = slpf_dfa_encode(state["host_cols"], state["host_text"], case["interval"])
            else:                                       # the file buffer archives are written to
                state["file"] = np.zeros(MIB + 4 * n, dtype=np.uint8)
    torch.cuda.synchronize()
    return state


def run(state):
    op = state["op"]
    if op == "parse":
        cols, status, _ = state["rx"].parse(state["text"], out=state.get("out"), status=state.get("status"),
                                            workspace=state.get("workspace"))
        return [cols, status]
    if op == "recognize":
        return [torch.cat([state["rx"].parse(x, recognize_only=True)[1] for x in state["texts"]])]
    if op == "serve":
        Batch(state["rxs"], [t.numel() for t in state["texts"]]).parse(state["texts"], outs=state["outs"],
                                                                       status=state["status"])
        return [state["arena"], state["status"]]
    if op == "batch":
        state["batch"].run()
        return [state["arena"], state["status"]]
    if op == "matches":
        pairs, total = state["rx"].matches(state["cols"], state["status"], state["n"], DNA_STOP_GROUP, state["kind"],
                                           cap=state["cap"])
        return [pairs, total]
    if op == "unarchive":
        return list(slpf_dfa_decode(state["archive"], state["text"], state["host_cols"].dtype.itemsize))
    archive = slpf_dfa_encode(state["host_cols"], state["host_text"], state["interval"])
    state["file"][:archive.size] = archive
    return [state["file"], archive.size]


def _col_bytes(pattern):
    rx = Regex(pattern, host_only=True)
    return rx.layout(1)[1]


def work(case):
    """Text read once, columns (matches: spans; archives: their sections) written once."""
    op = case["op"]
    if op in ("serve", "batch"):
        cb = [_col_bytes(_pattern_of(b)) for b in _bodies(case)]
        lens, which = _lengths(case)
        return {"bytes": float(sum(n + (n + 1) * cb[w] for n, w in zip(lens.tolist(), which))), "flops": 0.0}
    n = case["n"]
    cols = (n + 1) * _col_bytes(_pattern(case))
    if op == "recognize":
        total = 12 * n
    elif op == "matches":                                # 3 of 64 positions start a stop codon, 16 bytes a span
        total = cols + 16 * n * 3 // 64
    elif op in ("archive", "unarchive"):                 # the exceptions: 6 % of a log's columns, 24 % of a DNA text's
        total = n + cols + int(4 * n * (0.06 if case["re"] == "log" else 0.24))
    else:
        total = n + cols
    return {"bytes": float(total), "flops": 0.0}


def exact(case, seed):
    """Outputs are whole numbers (column ids, spans, bytes): compared for equality, nothing to round."""
    return None
