"""GPU parity of the two-cells-per-register kernel on 16 x 64 column tasks (tile 4x8v) for every
alignment type, and of the tile that a plan chooses by itself: which kernel a batch gets at the edges of
the rule, and that its scores are the oracle's there. Tolerance 0."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
PROT = synth.protein_scoring(99)
TYPES = {"global": (B.GLOBAL, None), "semiglobal": (B.SEMIGLOBAL, oracle.SEMIGLOBAL),
         "local": (B.LOCAL, oracle.LOCAL)}


def _plan(sc, flags=0, **env):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        return B.trioseq_plan(sc.alphabet, sc.sub, sc.gap, flags)
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def _strs(t, sc):
    return [synth.to_str(x, sc.alphabet) for x in t]


def _want(t, sc, kind):
    return oracle.align(*t, sc.sub, sc.gap) if kind is None else oracle.align_type(
        *t, sc.sub, sc.gap, kind)


def _rand(rng, shape, K):
    return tuple(rng.integers(0, K, size=n).astype(np.uint8) for n in shape)


@pytest.mark.parametrize("kind", TYPES)
@pytest.mark.parametrize("sc", [DNA, PROT], ids=["dna", "protein"])
def test_narrow_tile_exact(sc, kind):
    flags, okind = TYPES[kind]
    rng = np.random.default_rng(401)
    shapes = [(15, 15, 63), (16, 16, 64), (14, 14, 62), (17, 17, 65), (0, 0, 0), (1, 33, 2),
              (40, 0, 70), (0, 48, 130), (19, 31, 64), (20, 47, 128), (23, 64, 63), (130, 40, 90)]
    trips = [_rand(rng, s, len(sc.alphabet)) for s in shapes]
    trips.append(synth.related_triplet(402, 0, 300, sc, 0.1, 0.03, 3.0))  # several rebases
    plan = _plan(sc, flags, TRIOSEQ_SCORE_TILE="4x8v", TRIOSEQ_TEST_POISON=1)
    try:
        bt = B.trioseq_batch_create(plan, [_strs(t, sc) for t in trips])
        try:
            assert B.trioseq_batch_info(bt)["tile_label"] == "4x8v"
        finally:
            B.trioseq_batch_destroy(bt)
        got = B.trioseq_align_batch(plan, [_strs(t, sc) for t in trips]).tolist()
        assert got == [_want(t, sc, okind) for t in trips]
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("kind,mode,shapes,label", [
    ("global", B.SCORE_ONLY, [(90, 63, 127)], "8x8"),                  # 4 x 2 tasks: int32
    ("global", B.SCORE_ONLY, [(30, 64, 127)], "4x8v"),                 # 5 x 2
    ("global", B.WITH_TRACEBACK, [(30, 64, 63), (30, 47, 63)], "4x8"),  # 5 + 3 tasks: int32
    ("global", B.WITH_TRACEBACK, [(30, 64, 63), (30, 63, 63)], "4x8v"),
    ("local", B.SCORE_ONLY, [(30, 64, 127)], "4x8v"),
    ("semiglobal", B.SCORE_ONLY, [(9, 100, 100)] * 21, "4x8v"),        # 21 x 14 = 294 tasks
    ("semiglobal", B.SCORE_ONLY, [(9, 100, 100)] * 22, "8x8v"),        # 308: past two per SM (152)
    ("local", B.WITH_TRACEBACK, [(30, 64, 127)], "4x4"),               # no such keys: int32
    ("global", B.SCORE_ONLY, [(30, 64, 127), (20, 30, 40)], "4x4"),    # packs two triplets
], ids=str)
def test_default_tile(kind, mode, shapes, label):
    flags, okind = TYPES[kind]
    rng = np.random.default_rng(403)
    trips = [_rand(rng, s, 4) for s in shapes]
    plan = _plan(DNA, flags)
    try:
        strs = [_strs(t, DNA) for t in trips]
        bt = B.trioseq_batch_create(plan, strs, mode)
        try:
            assert B.trioseq_batch_info(bt)["tile_label"] == label
            B.trioseq_batch_run(bt)
            got = B.trioseq_batch_scores(bt, len(trips)).tolist()
        finally:
            B.trioseq_batch_destroy(bt)
        assert got == [_want(t, DNA, okind) for t in trips]
    finally:
        B.trioseq_plan_destroy(plan)
