"""GPU parity of the register-tiled affine kernel (affine.cu): shapes on both sides of its 16 x 32
column tasks, one and two triplets per register, chunked launches, and the plane kernel that takes
over when the boundary records exceed the memory budget. Tolerance 0."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()
PROT = synth.protein_scoring(77)
SHAPES = [(15, 15, 31), (16, 16, 32), (14, 14, 30), (17, 17, 33), (31, 47, 64), (1, 40, 2),
          (70, 1, 95), (0, 0, 33), (200, 40, 70), (33, 15, 63), (2, 33, 65)]


def _scores(sc, gap_open, trips, **env):
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        plan = B.trioseq_plan_affine(sc.alphabet, sc.sub, sc.gap, gap_open)
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v
    strs = [[synth.to_str(x, sc.alphabet) for x in t] for t in trips]
    try:
        bt = B.trioseq_batch_create(plan, strs)
        try:
            info = B.trioseq_batch_info(bt)
        finally:
            B.trioseq_batch_destroy(bt)
        return B.trioseq_align_batch(plan, strs).tolist(), info
    finally:
        B.trioseq_plan_destroy(plan)


@pytest.mark.parametrize("sc,gap_open,n,env,kernel,packing", [
    (DNA, -4, None, {}, "affine_kernel", 2),
    (PROT, -9, None, {}, "affine_kernel", 2),
    (DNA, -4, None, {"TRIOSEQ_PACKED": 0}, "affine_kernel", 1),
    (DNA, -1363, None, {}, "affine_kernel", 2),       # 12 |gamma| + 3 * 6 < 2^14: the largest opening that still packs ...
    (DNA, -1364, None, {}, "affine_kernel", 1),       # ... and the first that does not
    (DNA, -200000, None, {}, "affine_kernel", 1),
    (PROT, -9, 1, {}, "affine_kernel", 1),
    (DNA, -4, None, {"TRIOSEQ_SLAB_BUDGET_MB": 3}, "affine_kernel", 2),      # several chunks
    (PROT, -9, None, {"TRIOSEQ_SLAB_BUDGET_MB": 1}, "affine_plane_kernel", 1),
], ids=["dna", "protein", "unpacked", "bound", "past", "steep", "one", "chunks", "planes"])
def test_affine_wave_exact(sc, gap_open, n, env, kernel, packing):
    rng = np.random.default_rng(201)
    trips = [tuple(rng.integers(0, len(sc.alphabet), size=L).astype(np.uint8) for L in s)
             for s in SHAPES][:n]
    got, info = _scores(sc, gap_open, trips, TRIOSEQ_TEST_POISON=1, **env)
    assert (info["kernel"], info["packing"]) == (kernel, packing)
    assert got == [oracle.align_affine(*t, sc.sub, sc.gap, gap_open) for t in trips]
