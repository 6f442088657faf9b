"""Semi-global and local traceback on its default tile (4x4, records as readiness flags for batches too) and on 4x8
where the records would exceed the budget: scores, rows and spans equal the oracle's, on shapes at the edges
of 16 x 32 tasks and in a batch whose second run finds the records of the first."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
TYPES = {"semiglobal": (B.SEMIGLOBAL, oracle.SEMIGLOBAL), "local": (B.LOCAL, oracle.LOCAL)}


@pytest.mark.parametrize("kind", TYPES)
@pytest.mark.parametrize("budget_mb,tile", [(None, (4, 4)), (1, (4, 8))])
def test_typed_traceback_default_tile(kind, budget_mb, tile):
    flags, okind = TYPES[kind]
    rng = np.random.default_rng(741)
    shapes = [(0, 0, 0), (1, 1, 1), (20, 14, 30), (21, 15, 31), (22, 16, 32), (40, 47, 63), (40, 48, 64),
              (60, 70, 100), (0, 20, 40), (33, 0, 40), (90, 64, 33)]
    trips = [[rng.integers(0, 4, n).astype(np.uint8) for n in s] for s in shapes]
    trips.append(list(synth.related_triplet(742, 0, 110, DNA, 0.1, 0.03, 3.0)))
    if budget_mb:
        os.environ["TRIOSEQ_SLAB_BUDGET_MB"] = str(budget_mb)
    try:
        plan = B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap, flags)
    finally:
        os.environ.pop("TRIOSEQ_SLAB_BUDGET_MB", None)
    try:
        bt = B.trioseq_batch_create(plan, [[synth.to_str(s, DNA.alphabet) for s in t] for t in trips],
                                    B.WITH_TRACEBACK)
        try:
            assert B.trioseq_batch_info(bt)["tile"] == tile
            for _ in range(2):
                B.trioseq_batch_run(bt)
                got = B.trioseq_batch_scores(bt, len(trips)).tolist()
                for i, t in enumerate(trips):
                    score, rows, begin, end = oracle.align_type_tb(*t, DNA.sub, DNA.gap, okind)
                    text = tuple("".join("-" if v == 255 else DNA.alphabet[v] for v in r) for r in rows)
                    assert got[i] == score
                    assert B.trioseq_batch_alignment(bt, i) == text
                    assert B.trioseq_batch_span(bt, i) == (tuple(begin), tuple(end))
        finally:
            B.trioseq_batch_destroy(bt)
    finally:
        B.trioseq_plan_destroy(plan)
