"""A device without room for a batch's boundary records or codes, or for what comes after them: layouts that
need less answer, with the same results, before the call fails. The refused allocation is injected on the host
(TRIOSEQ_TEST_FAIL_ALLOC); nothing else changes on the device."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
# the allocations of a batch in their order: inputs, records, progress, scores, codes, rows
RECORDS, CODES, ROWS = 2, 5, 6


def _plan(fail, gap_open=None, flags=0, **env):
    env["TRIOSEQ_TEST_FAIL_ALLOC"] = fail
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        if gap_open is not None:
            return B.trioseq_plan_affine(DNA.alphabet, DNA.sub, DNA.gap, gap_open)
        return B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap, flags)
    finally:
        for k in env:
            os.environ.pop(k, None)


def _trips(shapes):
    rng = np.random.default_rng(831)
    return [tuple(rng.integers(0, 4, n).astype(np.uint8) for n in s) for s in shapes]


def _strs(trips):
    return [[synth.to_str(x, DNA.alphabet) for x in t] for t in trips]


def _info(plan, strs, mode):
    bt = B.trioseq_batch_create(plan, strs, mode)
    try:
        return B.trioseq_batch_info(bt)
    finally:
        B.trioseq_batch_destroy(bt)


@pytest.mark.parametrize("shapes,kernel,packing", [
    ([(200, 33, 40)], "affine_plane_kernel", 1),                 # one triplet: planes
    ([(60, 33, 40), (61, 40, 20), (9, 5, 70)], "affine_kernel", 2),  # several: a launch per pair
])
def test_affine(shapes, kernel, packing):
    trips = _trips(shapes)
    plan = _plan(1 + RECORDS, gap_open=-4)  # after the plan's own table of sigma
    try:
        info = _info(plan, _strs(trips), B.SCORE_ONLY)
        assert (info["kernel"], info["packing"]) == (kernel, packing)
    finally:
        B.trioseq_plan_destroy(plan)
    plan = _plan(1 + RECORDS, gap_open=-4)
    try:
        for _ in range(2):  # the second call has its room again
            got = B.trioseq_align_batch(plan, _strs(trips)).tolist()
            assert got == [oracle.align_affine(*t, DNA.sub, DNA.gap, -4) for t in trips]
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("flags,okind,label,fail", [
    (B.GLOBAL, oracle.GLOBAL, "4x8", RECORDS), (B.GLOBAL, oracle.GLOBAL, "4x8", CODES),
    (B.GLOBAL, oracle.GLOBAL, "4x8", ROWS), (B.LOCAL, oracle.LOCAL, "4x8", RECORDS)],
    ids=["records", "codes", "rows", "local"])
def test_rows(flags, okind, label, fail):
    # many more steps than slices (a = 3): the default tiles need more room than int32 4x8 here
    trips = _trips([(3, 40, 63)] * 9 + [(5, 33, 60)])
    plan = _plan(fail, flags=flags)
    try:
        assert _info(plan, _strs(trips), B.WITH_TRACEBACK)["tile_label"] == label
    finally:
        B.trioseq_plan_destroy(plan)
    plan = _plan(fail, flags=flags)
    try:
        got = B.trioseq_align_batch(plan, _strs(trips), B.WITH_TRACEBACK).tolist()
        for i, t in enumerate(trips):
            score, rows, _, _ = oracle.align_type_tb(*t, DNA.sub, DNA.gap, okind)
            assert got[i] == score
            assert B.trioseq_traceback(plan, i) == tuple(
                "".join("-" if v == 255 else DNA.alphabet[v] for v in r) for r in rows)
    finally:
        B.trioseq_plan_destroy(plan)


def test_pairs_and_nothing_smaller():
    trips = _trips([(3, 40, 40)] * 7)
    want = oracle.align_many(trips, DNA.sub, DNA.gap).tolist()
    plan = _plan(RECORDS)
    try:
        info = _info(plan, _strs(trips), B.SCORE_ONLY)
        assert (info["tile_label"], info["packing"]) == ("8x8", 2)
    finally:
        B.trioseq_plan_destroy(plan)
    plan = _plan(RECORDS, TRIOSEQ_SCORE_TILE="8x8")
    try:
        with pytest.raises(B.TrioseqError) as e:
            B.trioseq_align_batch(plan, _strs(trips))
        assert e.value.status == B.ENOMEM
        assert B.trioseq_align_batch(plan, _strs(trips)).tolist() == want
    finally:
        B.trioseq_plan_destroy(plan)
