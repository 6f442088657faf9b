"""GPU parity of the two-cells-per-register traceback kernel (wavefront_vl.cuh, tiles 8x8v
and 4x8v with traceback keys): scores and rows against the oracle on shapes at the edges of its 32 x 64 and
16 x 64 column tasks, on schemes at its sigma'' limit and one past it, and on triplets long enough to
rebase. Tolerance 0."""
import itertools
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
PROT = synth.protein_scoring(88)
TILES = ["8x8v", "4x8v"]


def _scheme(top):
    """Four letters, gap -10 (sigma'' = sub + 20), sigma'' from 0 to `top`."""
    sub = np.array([[top, 0, 3, 1], [0, top, 2, 7], [3, 2, top, 0], [1, 7, 0, 5]], dtype=np.int32) - 20
    return synth.Scoring("ACGT", sub, -10, np.full(4, 0.25), "edge")


def _plan(sc, **env):
    env = {"TRIOSEQ_TB_TILE": "8x8v", "TRIOSEQ_TEST_POISON": 1, **env}
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        return B.trioseq_plan(sc.alphabet, sc.sub, sc.gap)
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def _strs(t, sc):
    return [synth.to_str(x, sc.alphabet) for x in t]


def _check(plan, sc, trips, kernel=("wavefront_vl_kernel<8,4,0,traceback>",
                                     "wavefront_vl_kernel<4,4,0,traceback>")):
    strs = [_strs(t, sc) for t in trips]
    bt = B.trioseq_batch_create(plan, strs, B.WITH_TRACEBACK)
    try:
        assert B.trioseq_batch_info(bt)["kernel"] in kernel
    finally:
        B.trioseq_batch_destroy(bt)
    got = B.trioseq_align_batch(plan, strs, B.WITH_TRACEBACK)
    for i, t in enumerate(trips):
        score, rows = oracle.align(*t, sc.sub, sc.gap, traceback=True)
        assert int(got[i]) == score
        assert B.trioseq_traceback(plan, i) == tuple(
            "".join("-" if v == 255 else sc.alphabet[v] for v in r) for r in rows)


def _rand(rng, shape, K):
    return tuple(rng.integers(0, K, size=n).astype(np.uint8) for n in shape)


EDGES = [(31, 31, 63), (32, 32, 64), (30, 30, 62), (33, 33, 65), (1, 64, 128), (0, 40, 70),
         (70, 0, 65), (64, 31, 0), (5, 95, 1), (90, 100, 131), (150, 33, 60)]


@pytest.mark.parametrize("tile", TILES)
def test_tiny_shapes_one_batch(tile):
    rng = np.random.default_rng(301)
    plan = _plan(DNA, TRIOSEQ_TB_TILE=tile)
    try:
        _check(plan, DNA, [_rand(rng, s, 4) for s in itertools.product(range(4), repeat=3)])
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("sc", [DNA, PROT, _scheme(30)], ids=["dna", "protein", "limit"])
def test_tile_edges(sc, tile):
    rng = np.random.default_rng(302)
    plan = _plan(sc, TRIOSEQ_TB_TILE=tile)
    try:
        trips = [_rand(rng, s, len(sc.alphabet)) for s in EDGES]
        _check(plan, sc, trips)
        for t in trips[:4]:
            _check(plan, sc, [t])
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("sc", [DNA, PROT, _scheme(30)], ids=["dna", "protein", "limit"])
def test_rebasing_triplets(sc, tile):
    """Identical and related triplets of 260..420 residues: M' passes many rebases."""
    rng = np.random.default_rng(303)
    s = rng.integers(0, len(sc.alphabet), size=260).astype(np.uint8)
    s[:130] = np.argmax(np.diag(sc.sub))  # the steepest growth, then mixed
    plan = _plan(sc, TRIOSEQ_TB_TILE=tile)
    try:
        _check(plan, sc, [(s, s, s)])
        _check(plan, sc, [synth.related_triplet(304, 0, 420, sc, 0.15, 0.03, 3.0)])
        _check(plan, sc, [(s, s[:40], s[100:])])
    finally:
        B.trioseq_plan_destroy(plan)


def test_past_the_limit_runs_int32():
    rng = np.random.default_rng(305)
    sc = _scheme(31)
    plan = _plan(sc)
    try:
        _check(plan, sc, [_rand(rng, (40, 50, 70), 4)], ("wavefront_kernel<4,8,traceback,global>",))
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("L,sc", [(1000, DNA), (900, PROT)], ids=["dna", "protein"])
def test_long_triplets_equal_int32(L, sc, tile):
    t = _strs(synth.related_triplet(306, 0, L, sc, 0.1, 0.03, 3.0), sc)
    vl, ref = _plan(sc, TRIOSEQ_TB_TILE=tile), _plan(sc, TRIOSEQ_TB_TILE="4x8")
    try:
        got, want = (B.trioseq_align_batch(p, [t], B.WITH_TRACEBACK).tolist() for p in (vl, ref))
        assert got == want
        assert B.trioseq_traceback(vl, 0) == B.trioseq_traceback(ref, 0)
        assert B.trioseq_traceback_span(vl, 0) == B.trioseq_traceback_span(ref, 0)
    finally:
        B.trioseq_plan_destroy(vl)
        B.trioseq_plan_destroy(ref)
