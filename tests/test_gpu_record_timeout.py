"""Bounded waits on boundary records that are their own readiness flags, in the kernels with two values per
register. Under TRIOSEQ_TEST_NO_RECORDS a launch finds its first column task taken and its records released
but never written: the task's consumers get past their start and give up on the records, theirs on the records
of those. No wait lasts longer than 20 ms, the call reports ETIMEOUT, and the same process then aligns
exactly."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()


def _plan(flags, env):
    os.environ.update(env)
    try:
        return B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap, flags)
    finally:
        for k in env:
            os.environ.pop(k, None)


@pytest.mark.parametrize("flags,mode,shapes,tile,label", [
    (B.GLOBAL, B.SCORE_ONLY, [(40, 200, 300)], None, "4x8v"),
    (B.GLOBAL, B.SCORE_ONLY, [(40, 200, 300)], "8x8v", "8x8v"),
    (B.GLOBAL, B.SCORE_ONLY, [(40, 200, 300)], "8x16", "8x16"),
    (B.GLOBAL, B.WITH_TRACEBACK, [(40, 200, 300)], None, "4x8v"),
    (B.LOCAL, B.SCORE_ONLY, [(40, 200, 300)], "8x8v", "8x8v"),
    (B.GLOBAL, B.SCORE_ONLY, [(40, 223, 200)] * 40, None, "8x4"),
    (B.GLOBAL, B.SCORE_ONLY, [(40, 223, 200)] * 8, None, "4x4"),
], ids=["score", "wide", "widest", "rows", "local", "pairs", "few pairs"])
def test_records_that_never_come(flags, mode, shapes, tile, label):
    rng = np.random.default_rng(871)
    trips = [tuple(rng.integers(0, 4, L).astype(np.uint8) for L in s) for s in shapes]
    strs = [[synth.to_str(x, DNA.alphabet) for x in t] for t in trips]
    env = {"TRIOSEQ_SCORE_TILE": tile} if tile else {}
    plan = _plan(flags, {"TRIOSEQ_TEST_NO_RECORDS": "1", "TRIOSEQ_WAIT_MS": "20", **env})
    try:
        bt = B.trioseq_batch_create(plan, strs, mode)
        try:
            assert B.trioseq_batch_info(bt)["tile_label"] == label
        finally:
            B.trioseq_batch_destroy(bt)
        with pytest.raises(B.TrioseqError) as e:
            B.trioseq_align_batch(plan, strs, mode)
        assert e.value.status == B.ETIMEOUT
    finally:
        B.trioseq_plan_destroy(plan)
    plan = _plan(flags, env)
    try:
        got = B.trioseq_align_batch(plan, strs, mode).tolist()
    finally:
        B.trioseq_plan_destroy(plan)
    assert got[:2] == [oracle.align(*t, DNA.sub, DNA.gap) if flags == B.GLOBAL else
                       oracle.align_type(*t, DNA.sub, DNA.gap, oracle.LOCAL) for t in trips[:2]]
