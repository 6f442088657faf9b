"""GPU parity of the two forms of a step on 32 x 64 tasks (tile 8x8v): the residue ring of the local type at
slices around its block edges (refills at steps 16 modulo 32, blocks of 32), and the packed right columns of
the global score around a rebase (values rise 2048 above the base) and over several block columns. Scores are
integers and equal the oracle's."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
PROT = synth.protein_scoring(731)


@pytest.mark.parametrize("sc", [DNA, PROT], ids=["dna", "protein"])
@pytest.mark.parametrize("kind", ["global", "local"])
def test_slices_around_block_edges(kind, sc):
    rng = np.random.default_rng(732)
    trips = [[rng.integers(0, len(sc.alphabet), n).astype(np.uint8) for n in (a, b, c)]
             for a in (0, 1, 13, 14, 15, 16, 17, 18, 31, 32, 33, 47, 48, 49, 63, 64, 65, 96, 97, 130)
             for b, c in ((40, 70), (31, 64))]
    for a in (33, 64, 97):  # the best local alignment spans the blocks
        s = rng.integers(0, len(sc.alphabet), a).astype(np.uint8)
        trips.append([s, s, s])
    s = np.full(420, int(np.argmax(np.diag(sc.sub))), dtype=np.uint8)  # the steepest growth
    trips.append([s, s[:300], s[:200]])
    os.environ["TRIOSEQ_SCORE_TILE"] = "8x8v"
    try:
        plan = B.trioseq_plan(sc.alphabet, sc.sub, sc.gap, B.LOCAL if kind == "local" else B.GLOBAL)
    finally:
        del os.environ["TRIOSEQ_SCORE_TILE"]
    try:
        text = [[synth.to_str(s, sc.alphabet) for s in t] for t in trips]
        bt = B.trioseq_batch_create(plan, text)
        try:
            assert B.trioseq_batch_info(bt)["tile_label"] == "8x8v"
        finally:
            B.trioseq_batch_destroy(bt)
        got = B.trioseq_align_batch(plan, text).tolist()
    finally:
        B.trioseq_plan_destroy(plan)
    if kind == "local":
        want = [oracle.align_type(*t, sc.sub, sc.gap, oracle.LOCAL) for t in trips]
    else:
        want = oracle.align_many(trips, sc.sub, sc.gap).tolist()
    assert got == want
