"""A server's device-memory budget bounds what its launches take, for every kind of request whose tile a
launch chooses: affine gaps (records, or planes where the records exceed the budget), rows with short second
sequences (whose tile depends on the other requests of a launch) and scores that run in pairs. The device
memory taken while a burst is served stays within the budget, and every result is the plan's own."""
import time

import numpy as np
import pytest

from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DNA = synth.dna_scoring()
POOL = 192 << 20  # rounding of the stream-ordered pool (up to 32 MB for each large buffer of four slots)


def _serve(plan, trips, mode, budget):
    """Results of a burst, and the most device memory taken meanwhile."""
    free0 = torch.cuda.mem_get_info()[0]
    srv = B.trioseq_server_create([plan], hbm_budget=budget)
    got, least = {}, free0
    try:
        tickets = [B.trioseq_submit(srv, t, 0, mode)[1] for t in trips]
        t0 = time.time()
        while len(got) < len(tickets):
            for i, tk in enumerate(tickets):
                if i in got:
                    continue
                st, score, rows = B.trioseq_poll(srv, tk, sum(map(len, trips[i])) if mode else 0)
                if st == B.OK:
                    got[i] = (score, rows)
            least = min(least, torch.cuda.mem_get_info()[0])
            assert time.time() - t0 < 60
    finally:
        B.trioseq_server_destroy(srv)
    return [got[i] for i in range(len(trips))], free0 - least


@pytest.mark.parametrize("gap_open,mode,shape,n,budget", [
    (-4, B.SCORE_ONLY, (500, 500, 500), 12, 512 << 20),      # 328 MB of records each
    (-4, B.SCORE_ONLY, (500, 400, 400), 6, 128 << 20),       # 209 MB: over planes, 41 MB, one at a time
    (None, B.WITH_TRACEBACK, (300, 14, 63), 400, 64 << 20),  # 16 x 64 tasks alone, 32 x 64 among others
    (None, B.SCORE_ONLY, (300, 200, 200), 200, 64 << 20),    # pairs
], ids=["affine", "affine planes", "rows", "pairs"])
def test_budget_holds(gap_open, mode, shape, n, budget):
    torch.cuda.init()
    rng = np.random.default_rng(841)
    trips = [tuple(synth.to_str(rng.integers(0, 4, L).astype(np.uint8), DNA.alphabet) for L in shape)
             for _ in range(n)]
    if gap_open is None:
        plan = B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap)
    else:
        plan = B.trioseq_plan_affine(DNA.alphabet, DNA.sub, DNA.gap, gap_open)
    try:
        got, taken = _serve(plan, trips, mode, budget)
        assert taken <= budget + POOL
        want = B.trioseq_align_batch(plan, trips, mode).tolist()
        assert [s for s, _ in got] == want
        if mode:
            assert [r for _, r in got] == [B.trioseq_traceback(plan, i) for i in range(n)]
    finally:
        B.trioseq_plan_destroy(plan)
