"""GPU parity of the two-triplets-per-register kernel (tiles 8x8, 8x4, 4x8, 4x4) where it can go wrong:
lengths at the edges of column tasks and of the residue ring's blocks, pairs of unequal lengths, a triplet
paired with itself, empty sequences, alphabets with and without repeated profiles, and the tile rule. Scores
are integers and equal the oracle's."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
PROT = synth.protein_scoring(701)


def _plan(sc, **env):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        return B.trioseq_plan(sc.alphabet, sc.sub, sc.gap)
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v


def _check(sc, trips, tile=None, **env):
    plan = _plan(sc, **({"TRIOSEQ_SCORE_TILE": tile} if tile else {}), **env)
    try:
        bt = B.trioseq_batch_create(plan, [[synth.to_str(s, sc.alphabet) for s in t] for t in trips])
        try:
            info = B.trioseq_batch_info(bt)
            assert info["kernel"].startswith("wavefront_vp_kernel") and info["packing"] == 2, info
            for _ in range(2):  # the records of the first run must not show in the second
                B.trioseq_batch_run(bt)
                got = B.trioseq_batch_scores(bt, len(trips)).tolist()
                assert got == oracle.align_many(trips, sc.sub, sc.gap).tolist()
        finally:
            B.trioseq_batch_destroy(bt)
        return info["tile"]
    finally:
        B.trioseq_plan_destroy(plan)


def _rand(rng, lens, K):
    return [rng.integers(0, K, n).astype(np.uint8) for n in lens]


@pytest.mark.parametrize("tile", ["8x8", "8x4", "4x8", "4x4"])
@pytest.mark.parametrize("sc", [DNA, PROT], ids=["dna", "protein"])
def test_edges(tile, sc):
    rng = np.random.default_rng(702)
    shapes = [(0, 0, 0), (0, 5, 9), (9, 0, 40), (1, 1, 1), (10, 31, 32), (11, 32, 31), (12, 15, 63),
              (13, 16, 64), (15, 63, 31), (16, 64, 33), (17, 33, 65), (30, 95, 96), (31, 96, 95),
              (32, 47, 48), (33, 48, 47), (47, 64, 64), (48, 70, 90), (49, 31, 33), (63, 64, 65),
              (64, 30, 30), (65, 31, 31), (95, 33, 70), (97, 70, 33), (150, 40, 66), (20, 66, 40)]
    trips = [_rand(rng, s, len(sc.alphabet)) for s in shapes]
    assert len(trips) % 2  # the last unit pairs a triplet with itself
    _check(sc, trips, tile)


@pytest.mark.parametrize("tile", ["8x4", "4x4"])
@pytest.mark.parametrize("K", [2, 15, 16, 32])  # both profile layouts, the largest alphabet
def test_alphabets(tile, K):
    rng = np.random.default_rng(703 + K)
    sub = rng.integers(-4, 5, (K, K))
    sub = np.tril(sub) + np.tril(sub, -1).T
    sc = synth.Scoring("ABCDEFGHIJKLMNOPQRSTUVWXYZabcdef"[:K], sub.astype(np.int32), -3, np.full(K, 1.0 / K))
    shapes = [(90, 70, 61), (14, 77, 80), (91, 66, 64), (33, 100, 35)]
    _check(sc, [_rand(rng, s, K) for s in shapes], tile)


@pytest.mark.parametrize("n,lo,hi,tile", [(8, 100, 200, (4, 4)),    # at most two tasks per SM
                                          (200, 100, 200, (8, 4)),
                                          (600, 34, 46, (4, 4))])   # 16 x 32 tasks pad less
def test_tile_rule(n, lo, hi, tile):
    w = synth.config2(seed=704, n=n, lo=lo, hi=hi)
    assert _check(DNA, w.triplets) == tile


def test_tile_rule_over_the_record_budget():
    w = synth.config2(seed=705, n=40, lo=100, hi=200)
    assert _check(DNA, w.triplets, TRIOSEQ_SLAB_BUDGET_MB=1) == (8, 8)
