"""The autotuner measures what an untuned plan takes as well, so that tuning does not lose to it: pairs of
triplets that run on the 8x4 tile (10% faster than any of the other tiles on this batch) keep it, triplets
that fit no 16-bit half are tuned over what can take them, and results stay the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()


def _kernel(plan, strs):
    """(tile label, best kernel ms of six runs, scores)"""
    bt = B.trioseq_batch_create(plan, strs)
    try:
        B.trioseq_batch_profile(bt)
        ms = []
        for _ in range(6):
            B.trioseq_batch_run(bt)
            got = B.trioseq_batch_scores(bt, len(strs))
            ms.append(B.trioseq_batch_timing(bt)[0])
        return B.trioseq_batch_info(bt)["tile_label"], min(ms), got
    finally:
        B.trioseq_batch_destroy(bt)


def test_tuned_pairs_are_not_slower():
    rng = np.random.default_rng(861)
    trips = [tuple(rng.integers(0, 4, L).astype(np.uint8) for L in (250, 255, 31)) for _ in range(2000)]
    strs = [[synth.to_str(x, DNA.alphabet) for x in t] for t in trips]
    plan, tuned = (B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap) for _ in range(2))
    try:
        choice = B.trioseq_plan_autotune(tuned, strs, B.SCORE_ONLY)
        label, ms, want = _kernel(plan, strs)
        _, tuned_ms, got = _kernel(tuned, strs)
        assert label == "8x4" and choice["tile"] == (8, 4)
        assert tuned_ms < 1.05 * ms
        assert got.tolist() == want.tolist()
        assert got[:8].tolist() == oracle.align_many(trips[:8], DNA.sub, DNA.gap).tolist()
        # a scheme under which such lengths fit no 16-bit half, with negative sigma''
        long = [tuple(rng.integers(0, 4, L).astype(np.uint8) for L in (250, 250, 250)) for _ in range(2)]
        neg = synth.Scoring("ACGT", DNA.sub * 12, DNA.gap, DNA.freqs, "steep")
        steep = B.trioseq_plan(neg.alphabet, neg.sub, neg.gap)
        try:
            ls = [[synth.to_str(x, DNA.alphabet) for x in t] for t in long]
            B.trioseq_plan_autotune(steep, ls, B.SCORE_ONLY)
            assert B.trioseq_align_batch(steep, ls).tolist() == \
                oracle.align_many(long, neg.sub, neg.gap).tolist()
        finally:
            B.trioseq_plan_destroy(steep)
    finally:
        B.trioseq_plan_destroy(plan)
        B.trioseq_plan_destroy(tuned)
