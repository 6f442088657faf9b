"""GPU parity of the traceback walk on long runs of gaps along the third sequence, which tiles of 4 lane
columns probe straight from the codes, 32 cells at a time: runs that end inside a tube, within a probe and at
its edges, followed by matches and by other moves, at the ends of the cube too. Rows, scores and
spans equal the oracle's."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
TYPES = {"global": (B.GLOBAL, oracle.GLOBAL), "semiglobal": (B.SEMIGLOBAL, oracle.SEMIGLOBAL),
         "local": (B.LOCAL, oracle.LOCAL)}


def _triplets():
    rng = np.random.default_rng(811)

    def rnd(n):
        return rng.integers(0, 4, size=n).astype(np.uint8)

    out = [(rnd(3), rnd(4), rnd(400)), (rnd(0), rnd(0), rnd(97)), (rnd(18), rnd(17), rnd(230))]
    for gap in (4, 8, 15, 16, 40, 41, 44, 45, 64, 88, 130):  # one insertion in S2 between matches
        core = rnd(70)
        at = int(rng.integers(20, 50))
        out.append((core, core.copy(), np.concatenate([core[:at], rnd(gap), core[at:]])))
    core = rnd(60)  # several insertions, and one in each of the other sequences
    out.append((np.concatenate([core[:30], rnd(25), core[30:]]), np.concatenate([core[:12], rnd(33), core[12:]]),
                np.concatenate([rnd(50), core[:20], rnd(47), core[20:41], rnd(60), core[41:], rnd(90)])))
    return out


@pytest.mark.parametrize("kind,tile", [
    ("global", None), ("global", "4x8v"), ("global", "8x8v"), ("global", "4x4"), ("global", "8x4"),
    ("global", "4x8"), ("global", "8x8"), ("semiglobal", None), ("local", None)], ids=str)
def test_gap_runs(kind, tile):
    flags, okind = TYPES[kind]
    if tile:
        os.environ["TRIOSEQ_TB_TILE"] = tile
    try:
        plan = B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap, flags)
    finally:
        os.environ.pop("TRIOSEQ_TB_TILE", None)
    trips = _triplets()
    try:
        got = B.trioseq_align_batch(plan, [[synth.to_str(s, DNA.alphabet) for s in t] for t in trips],
                                    B.WITH_TRACEBACK).tolist()
        for i, t in enumerate(trips):
            score, rows, begin, end = oracle.align_type_tb(*t, DNA.sub, DNA.gap, okind)
            assert got[i] == score
            assert B.trioseq_traceback(plan, i) == tuple(
                "".join("-" if v == 255 else DNA.alphabet[v] for v in r) for r in rows)
            assert B.trioseq_traceback_span(plan, i) == (tuple(begin), tuple(end))
    finally:
        B.trioseq_plan_destroy(plan)
