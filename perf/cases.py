"""What users of the engine have it do, as cases to be timed and compared.

A case is one call of the public binding (paper_2605_28400_gb300.binding) on seeded synthetic
triplets: one triplet or a batch, score only or with the aligned rows, every alignment type, the
linear and the affine gap model, DNA and protein scoring, through the per-call entry, a
device-resident batch, the allocation-free entry or the server. Plans are made with their defaults,
as the quick start does; nothing is autotuned.
"""
from __future__ import annotations

import ctypes
import itertools
import math

import numpy as np
import torch

from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

TYPES = {"global": B.GLOBAL, "semiglobal": B.SEMIGLOBAL, "local": B.LOCAL}
GAP_OPEN = -4  # affine cases: the opening of the benchmark's affine line


def _case(path, alphabet, n, lo, hi, traceback=False, kind="global", affine=False, related=True):
    """path: align (host strings in, scores and rows out), resident (a device-resident batch, run
    and read), noalloc (device pointers) or server (submit all, poll all). Ancestors are lo..hi
    residues long; `related` triplets descend from one ancestor, others are three independent
    sequences of lo..hi residues each."""
    return {"path": path, "alphabet": alphabet, "n": n, "lo": lo, "hi": hi, "traceback": traceback,
            "type": kind, "affine": affine, "related": related}


def listed():
    return [
        # the smallest call: one short DNA triplet already on the device, score only, from a
        # program that must not allocate
        {"name": "noalloc_dna100", **_case("noalloc", "dna", 1, 100, 100)},
        # an interactive request: one 128-residue DNA triplet, score and aligned rows
        {"name": "dna128_rows", **_case("align", "dna", 1, 128, 128, traceback=True, related=False)},
        # one protein family of the usual length, score only (the serving stream's median length)
        {"name": "protein300_score", **_case("align", "protein", 1, 300, 300)},
        # one gene-length DNA triplet, score and rows
        {"name": "dna1000_rows", **_case("align", "dna", 1, 1000, 1000, traceback=True)},
        # the longest alignment that still keeps its whole code cube on the card with room to spare
        {"name": "dna3000_rows", **_case("align", "dna", 1, 3000, 3000, traceback=True)},
        # the largest single triplet, score only, device resident (the benchmark's main line)
        {"name": "protein4000_score", **_case("resident", "protein", 1, 4000, 4000)},
        # best local score of one long protein triplet
        {"name": "protein1500_local", **_case("align", "protein", 1, 1500, 1500, kind="local")},
        # guide-tree scoring: thousands of short DNA triplets in one call
        {"name": "dna_batch4096_score", **_case("align", "dna", 4096, 100, 300)},
        # reads against reads: overlaps of short DNA triplets
        {"name": "dna_batch1024_semiglobal", **_case("align", "dna", 1024, 100, 300, kind="semiglobal")},
        # a set of gene fragments whose alignments are all wanted
        {"name": "dna_batch96_rows", **_case("align", "dna", 96, 200, 600, traceback=True)},
        # affine gaps over a batch of short DNA triplets
        {"name": "dna_batch256_affine", **_case("align", "dna", 256, 100, 300, affine=True)},
        # a burst on the server: DNA and protein, a fifth with rows, lognormal lengths to 2,000
        {"name": "server_mix300", **_case("server", "mixed", 300, 50, 2000)},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges, its sizes spread over their logarithm."""
    alphabet = rng.choice(["dna", "dna", "protein"])
    kind = rng.choice(["global", "global", "semiglobal", "local"])
    what = rng.choice(["score", "score", "rows", "rows", "batch", "batch", "batch_rows", "noalloc",
                       "affine", "server"])
    if what == "score":
        L = _log(rng, 30, 4000 if kind == "global" else 3000)
        return _case(rng.choice(["align", "resident"]), alphabet, 1, L, L, kind=kind)
    if what == "rows":
        L = _log(rng, 30, 3000 if kind == "global" else 2000)
        return _case("align", alphabet, 1, L, L, traceback=True, kind=kind)
    if what == "batch":  # at most the cells of 4,096 triplets of 100..300 residues
        hi = _log(rng, 60, 600)
        lo = max(20, int(hi * rng.uniform(0.2, 1.0)))
        n = _log(rng, 2, min(4096, int(2.5e10 / (0.5 * (lo + hi)) ** 3)))
        return _case(rng.choice(["align", "align", "resident"]), alphabet, n, lo, hi, kind=kind,
                     related=rng.random() < 0.7)
    if what == "batch_rows":
        hi = _log(rng, 40, 600)
        lo = max(20, int(hi * rng.uniform(0.2, 1.0)))
        return _case("align", alphabet, _log(rng, 2, 96), lo, hi, traceback=True, kind=kind,
                     related=rng.random() < 0.7)
    if what == "noalloc":
        L = _log(rng, 20, 400)
        return _case("noalloc", alphabet, 1, L, L)
    if what == "affine":
        hi = _log(rng, 40, 300)
        return _case("align", alphabet, _log(rng, 1, 256), max(20, int(hi * rng.uniform(0.3, 1.0))),
                     hi, affine=True)
    return _case("server", "mixed", _log(rng, 20, 300), 50, _log(rng, 200, 2000))


def _scoring(alphabet):
    return synth.dna_scoring() if alphabet == "dna" else synth.protein_scoring(1003)


def _triplet(seed, idx, L, sc, related, lo, hi):
    if related:
        rates = (0.05, 0.02, 2.0) if sc.name == "dna" else (0.15, 0.03, 3.0)
        return synth.related_triplet(seed, idx, L, sc, *rates)
    lens = lo + synth.draws_u64(synth.stream_key(seed, idx, 0x1E), np.arange(3)) % np.uint64(hi - lo + 1)
    return tuple(synth.random_seq(synth.stream_key(seed, idx, q), int(lens[q]), sc.freqs)
                 for q in range(3))


def _lengths(case, seed):
    lo, hi, n = case["lo"], case["hi"], case["n"]
    return lo + (synth.draws_u64(synth.stream_key(seed, 0xB), np.arange(n)) %
                 np.uint64(hi - lo + 1)).astype(np.int64)


def _triplets(case, seed):
    sc = _scoring(case["alphabet"])
    return sc, [_triplet(seed, i, int(L), sc, case["related"], case["lo"], case["hi"])
                for i, L in enumerate(_lengths(case, seed))]


class State:
    """What the calling program keeps: its inputs and the handles it made."""

    def __init__(self):
        self.plans, self.batch, self.server = [], None, None

    def __del__(self):
        if self.server is not None:
            B.trioseq_server_destroy(self.server)
        if self.batch is not None:
            B.trioseq_batch_destroy(self.batch)
        for p in self.plans:
            B.trioseq_plan_destroy(p)


def prepare(case, seed):
    torch.cuda.init()
    s = State()
    s.case = case
    s.mode = B.WITH_TRACEBACK if case["traceback"] else B.SCORE_ONLY
    if case["path"] == "server":
        dna, prot, reqs = synth.config4(seed, case["n"], case["lo"], case["hi"])
        s.plans = [B.trioseq_plan(x.alphabet, x.sub, x.gap) for x in (dna, prot)]
        s.reqs = [(tuple(synth.to_str(c, (prot if r["protein"] else dna).alphabet)
                         for c in r["triplet"]), int(r["protein"]),
                   B.WITH_TRACEBACK if r["traceback"] else B.SCORE_ONLY) for r in reqs]
        s.server = B.trioseq_server_create(s.plans, 8 << 30)  # a service's share of the card
        return s
    s.sc, codes = _triplets(case, seed)
    if case["path"] == "noalloc":
        text = np.frombuffer(s.sc.alphabet.encode(), dtype=np.uint8)
        s.dev = [torch.from_numpy(text[c].copy()).cuda() for c in codes[0]]
        s.out = torch.zeros(1, dtype=torch.int32, device="cuda")
        return s
    s.triplets = [tuple(synth.to_str(c, s.sc.alphabet) for c in t) for t in codes]
    if case["affine"]:
        s.plans = [B.trioseq_plan_affine(s.sc.alphabet, s.sc.sub, s.sc.gap, GAP_OPEN)]
    else:
        s.plans = [B.trioseq_plan(s.sc.alphabet, s.sc.sub, s.sc.gap, TYPES[case["type"]])]
    if case["path"] == "resident":
        s.batch = B.trioseq_batch_create(s.plans[0], s.triplets, s.mode)
    return s


def _bytes(rows, case):
    """All aligned rows one after another, in an array whose size the case alone gives."""
    out = np.zeros(case["n"] * 3 * (case["hi"] if case["path"] == "server" else 4 * case["hi"] + 100),
                   dtype=np.uint8)
    text = np.frombuffer("".join(itertools.chain.from_iterable(rows)).encode(), dtype=np.uint8)
    out[:text.size] = text
    return out


def run(s):
    path = s.case["path"]
    if path == "noalloc":
        a, b, c = s.dev
        st = B.trioseq_align_noalloc(s.sc.alphabet, s.sc.sub, s.sc.gap, a.data_ptr(), a.numel(),
                                     b.data_ptr(), b.numel(), c.data_ptr(), c.numel(),
                                     s.out.data_ptr(), torch.cuda.current_stream())
        if st != B.OK:
            raise RuntimeError(B.trioseq_strerror(st))
        return s.out
    if path == "server":
        tickets = [B.trioseq_submit(s.server, t, pid, mode)[1] for t, pid, mode in s.reqs]
        scores = np.zeros(len(tickets), dtype=np.int32)
        rows = [()] * len(tickets)
        waiting = list(range(len(tickets)))
        while waiting:
            left = []
            for q in waiting:
                t, _, mode = s.reqs[q]
                cap = sum(map(len, t)) if mode == B.WITH_TRACEBACK else 0
                st, score, got = B.trioseq_poll(s.server, tickets[q], cap)
                if st == B.EAGAIN:
                    left.append(q)
                    continue
                scores[q], rows[q] = score, got or ()
            waiting = left
        return {"scores": scores, "rows": _bytes(rows, s.case)}
    stream = torch.cuda.current_stream()
    if path == "resident":
        B.trioseq_batch_run(s.batch, stream)
        return {"scores": B.trioseq_batch_scores(s.batch, len(s.triplets), stream)}
    scores = B.trioseq_align_batch(s.plans[0], s.triplets, s.mode, stream)
    if s.mode == B.SCORE_ONLY:
        return {"scores": scores}
    rows = [B.trioseq_traceback(s.plans[0], i) for i in range(len(s.triplets))]
    return {"scores": scores, "rows": _bytes(rows, s.case)}


def work(case):
    """Every residue read once, every score and row written once; per cell of the cube the
    recurrence's 7 additions and 6 maxima (affine: one addition and one maximum for each of its 7
    moves from 13 states)."""
    if case["path"] == "server":  # lognormal lengths about 300, clipped
        z = np.linspace(-3, 3, 601)
        w = np.exp(-z * z / 2)
        L = np.clip(300.0 * np.exp(0.8 * z), case["lo"], case["hi"])
        residues, cells = 3 * float((L * w).sum() / w.sum()), float((L ** 3 * w).sum() / w.sum())
        residues, cells, rows = residues * case["n"], cells * case["n"], 0.2  # a fifth with rows
    else:
        L = np.linspace(case["lo"], case["hi"], 201)
        residues, cells = 3 * float(L.mean()) * case["n"], float((L ** 3).mean()) * case["n"]
        if not case["related"]:
            cells = float(L.mean()) ** 3 * case["n"]
        rows = 1.0 if case["traceback"] else 0.0
    return {"bytes": residues * (1 + rows * 1.05) + 4.0 * case["n"],
            "flops": cells * (182 if case["affine"] else 13)}


# ---- the same results in 64-bit torch -----------------------------------------------------------

_MOVES = [m for m in itertools.product((1, 0), repeat=3) if any(m)]
_NEG = -(1 << 50)


def _planes(codes, sub, gap, kind, gap_open):
    """Scores of a list of triplets by the recurrence itself, plane i + j + k after plane."""
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    n = len(codes)
    a, b, c = (torch.tensor([len(t[q]) for t in codes], device=dev).view(n, 1, 1) for q in range(3))
    A, Bm, C = int(a.max()), int(b.max()), int(c.max())
    K = sub.shape[0]
    sub = torch.as_tensor(np.asarray(sub), dtype=torch.int64, device=dev).reshape(-1)

    def padded(q, size):  # residue of index 1.. at its index
        out = torch.zeros((n, size + 1), dtype=torch.int64)
        for t, x in enumerate(codes):
            out[t, 1:len(x[q]) + 1] = torch.from_numpy(np.asarray(x[q], dtype=np.int64))
        return out.to(dev)

    X, Y, Z = padded(0, A), padded(1, Bm).view(n, -1, 1), padded(2, C).view(n, 1, -1)
    j = torch.arange(Bm + 1, device=dev).view(1, -1, 1)
    k = torch.arange(C + 1, device=dev).view(1, 1, -1)
    yz = sub[Y * K + Z]
    states = [(0, 0, 0)]
    if gap_open is not None:  # per pair: 0 both residues, 1 gap in its first, 2 in its second
        for _ in range(3):
            states = sorted({tuple(_kinds(m, s)[0]) for m in _MOVES for s in states} | set(states))
    S = len(states)
    index = {s: e for e, s in enumerate(states)}
    full = lambda: torch.full((S, n, Bm + 2, C + 2), _NEG, dtype=torch.int64, device=dev)  # noqa: E731
    past = [full() for _ in range(4)]
    best = torch.full((n, 1, 1), _NEG, dtype=torch.int64, device=dev)
    for d in range(A + Bm + C + 1):
        cur = past[d & 3]
        cur.fill_(_NEG)
        i = d - j - k
        inside = (i >= 0) & (i <= a) & (j <= b) & (k <= c)
        x = torch.gather(X, 1, i.clamp(0, A).expand(n, -1, -1).reshape(n, -1)).view(n, Bm + 1, C + 1)
        xy, xz = sub[x * K + Y], sub[x * K + Z]
        val = cur[:, :, 1:, 1:]
        for m in _MOVES:
            di, dj, dk = m
            cost = (xy if di and dj else gap * (di + dj)) + (xz if di and dk else gap * (di + dk)) \
                + (yz if dj and dk else gap * (dj + dk))
            src = past[(d - di - dj - dk) & 3]
            src = src[:, :, 1 - dj:Bm + 2 - dj, 1 - dk:C + 2 - dk]
            for e, s in enumerate(states):
                to, opened = _kinds(m, s) if gap_open is not None else ((0, 0, 0), 0)
                cand = src[e] + cost + (gap_open * opened if gap_open is not None else 0)
                torch.maximum(val[index[tuple(to)]], cand, out=val[index[tuple(to)]])
        axis = ((i == 0).long() + (j == 0) + (k == 0)) >= 2
        if d == 0 or kind != "global":
            val[0] = torch.where(axis if kind != "global" else axis & (d == 0), 0, val[0])
        if kind == "local":
            val.clamp_(min=0)
        val.masked_fill_(~inside, _NEG)
        counts = inside if kind == "local" else inside & (
            (i == a) & (j == b) & (k == c) if kind == "global" else (i == a) | (j == b) | (k == c))
        here = torch.where(counts, val.amax(dim=0), _NEG)
        best = torch.maximum(best, here.amax(dim=(1, 2), keepdim=True))
    return best.view(n)


def _kinds(m, s):
    """The pairs' kinds after move m from kinds s, and the gap runs it opens."""
    to, opened = list(s), 0
    for pair, (p, q) in enumerate(((0, 1), (0, 2), (1, 2))):
        if m[p] and m[q]:
            to[pair] = 0
        elif m[p] or m[q]:
            now = 2 if m[p] else 1
            opened += s[pair] != now
            to[pair] = now
    return to, opened


def exact(case, seed):
    if case["path"] == "server":
        return None  # a mix of sizes and schemes: minutes
    lengths = _lengths(case, seed)
    cost = float((lengths.astype(float) ** 3).sum()) * (20 if case["affine"] else 1)
    if cost > 3e9:
        return None  # too long in 64 bits
    sc, codes = _triplets(case, seed)
    out = torch.zeros(len(codes), dtype=torch.int64)
    order = sorted(range(len(codes)), key=lambda t: -max(map(len, codes[t])))
    step = max(1, int(6e7 / (13 if case["affine"] else 1) / (max(map(len, codes[order[0]])) + 2) ** 2))
    for at in range(0, len(order), step):
        part = order[at:at + step]
        out[part] = _planes([codes[t] for t in part], sc.sub, sc.gap, case["type"],
                            GAP_OPEN if case["affine"] else None).cpu()
    if case["path"] == "noalloc":
        return out
    return {"scores": out, "rows": None} if case["traceback"] else {"scores": out}
