"""Where the results of trioseq_align_batch pass the host: through pinned memory behind the inputs, directly
when no pinned room is left for them (the refusal is injected on the host, TRIOSEQ_TEST_FAIL_PINNED) and
directly when they exceed 16 MB; a server's slots reserve none. Results equal the oracle's."""
import os

import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu

DNA = synth.dna_scoring()


def _text(rows):
    return tuple("".join("-" if v == 255 else DNA.alphabet[v] for v in r) for r in rows)


def _trips(shape, n):
    rng = np.random.default_rng(851)
    return [tuple(rng.integers(0, 4, L).astype(np.uint8) for L in shape) for _ in range(n)]


def _plan(fail=0):
    os.environ["TRIOSEQ_TEST_FAIL_PINNED"] = str(fail)
    try:
        return B.trioseq_plan(DNA.alphabet, DNA.sub, DNA.gap)
    finally:
        del os.environ["TRIOSEQ_TEST_FAIL_PINNED"]


def _check(plan, trips, sample):
    strs = [[synth.to_str(x, DNA.alphabet) for x in t] for t in trips]
    got = B.trioseq_align_batch(plan, strs, B.WITH_TRACEBACK)
    for i in sample:
        score, rows = oracle.align(*trips[i], DNA.sub, DNA.gap, traceback=True)
        assert int(got[i]) == score
        assert B.trioseq_traceback(plan, i) == _text(rows)


def test_no_pinned_room_for_results():
    trips = _trips((40, 35, 50), 5)
    plan = _plan(1)  # the first pinned allocation: inputs and results together
    try:
        for _ in range(2):
            _check(plan, trips, range(5))
    finally:
        B.trioseq_plan_destroy(plan)


def test_results_beyond_the_staging_limit():
    trips = _trips((1, 2, 3000), 1900)  # 3 x 3,003 bytes each: 17 MB of rows
    plan = _plan()
    try:
        _check(plan, trips, (0, 1, 950, 1899))
    finally:
        B.trioseq_plan_destroy(plan)


def test_server_slot_takes_two_pinned_buffers():
    """Inputs, then results of its own: a third allocation of the launch never comes."""
    t = _trips((40, 35, 50), 1)[0]
    plan = _plan(3)
    srv = B.trioseq_server_create([plan])
    try:
        _, ticket = B.trioseq_submit(srv, [synth.to_str(x, DNA.alphabet) for x in t], 0, B.WITH_TRACEBACK)
        st = B.EAGAIN
        while st == B.EAGAIN:
            st, score, rows = B.trioseq_poll(srv, ticket, 200)
        want, wrows = oracle.align(*t, DNA.sub, DNA.gap, traceback=True)
        assert (score, rows) == (want, _text(wrows))
    finally:
        B.trioseq_server_destroy(srv)
        B.trioseq_plan_destroy(plan)
