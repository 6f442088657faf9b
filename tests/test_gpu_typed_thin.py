"""GPU parity of semi-global and local traceback where the third sequence is by far the longest: one such
triplet runs on 16 x 64 column tasks, every other one and every batch on 16 x 32. The tile on both sides of
the line, and scores, rows and spans against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
TYPES = {"semiglobal": (B.SEMIGLOBAL, oracle.SEMIGLOBAL), "local": (B.LOCAL, oracle.LOCAL)}


@pytest.mark.parametrize("kind", TYPES)
@pytest.mark.parametrize("shapes,tile", [
    ([(20, 60, 240)], (4, 8)), ([(20, 60, 239)], (4, 4)), ([(20, 61, 240)], (4, 4)),
    ([(0, 0, 130)], (4, 8)), ([(0, 0, 0)], (4, 4)), ([(10, 3, 400)], (4, 8)),
    ([(10, 3, 400), (3, 10, 300)], (4, 4)), ([(240, 20, 60)], (4, 4)), ([(20, 240, 60)], (4, 4))], ids=str)
def test_tile_and_rows(kind, shapes, tile):
    flags, okind = TYPES[kind]
    rng = np.random.default_rng(821)
    trips = [[rng.integers(0, 4, n).astype(np.uint8) for n in s] for s in shapes]
    plan = B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap, flags)
    try:
        bt = B.trioseq_batch_create(plan, [[synth.to_str(s, DNA.alphabet) for s in t] for t in trips],
                                    B.WITH_TRACEBACK)
        try:
            assert B.trioseq_batch_info(bt)["tile"] == tile
            B.trioseq_batch_run(bt)
            got = B.trioseq_batch_scores(bt, len(trips)).tolist()
            for i, t in enumerate(trips):
                score, rows, begin, end = oracle.align_type_tb(*t, DNA.sub, DNA.gap, okind)
                assert got[i] == score
                assert B.trioseq_batch_alignment(bt, i) == tuple(
                    "".join("-" if v == 255 else DNA.alphabet[v] for v in r) for r in rows)
                assert B.trioseq_batch_span(bt, i) == (tuple(begin), tuple(end))
        finally:
            B.trioseq_batch_destroy(bt)
    finally:
        B.trioseq_plan_destroy(plan)
