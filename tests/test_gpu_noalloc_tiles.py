"""trioseq_align_noalloc where its choice of tile changes: 16 x 64 and 32 x 64 tasks of two cells per register,
and int32 where the records of those exceed the scratch or the scheme is past their range (a negative
sigma'', a sigma'' above 33). Scores are integers and equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2605_28400_gb300 import binding as B
from paper_2605_28400_gb300 import synth

pytestmark = pytest.mark.gpu


def _scheme(match, mismatch, gap):
    sub = np.full((4, 4), mismatch, dtype=np.int32)
    np.fill_diagonal(sub, match)
    return synth.Scoring("ACGT", sub, gap, np.full(4, 0.25))


DNA = synth.dna_scoring()


@pytest.mark.parametrize("sc,shape", [
    (DNA, (40, 607, 511)),                 # 38 x 8 = 304 tasks: two per SM on 152
    (DNA, (40, 608, 511)),                 # 39 x 8: 32 x 64 tasks
    (DNA, (3, 4000, 4000)),                # 32 x 64 tasks fit
    (DNA, (3, 5000, 5000)),                # only the int32 records fit
    (_scheme(2, -1, 0), (60, 70, 80)),     # sigma'' = -1
    (_scheme(13, -1, -10), (60, 70, 80)),  # sigma'' = 33
    (_scheme(14, -1, -10), (60, 70, 80)),  # sigma'' = 34
], ids=str)
def test_noalloc_tiles(sc, shape):
    torch = pytest.importorskip("torch")
    torch.cuda.set_device(0)
    rng = np.random.default_rng(721)
    trip = [rng.integers(0, 4, n).astype(np.uint8) for n in shape]
    dev = [torch.from_numpy(np.frombuffer(synth.to_str(s, sc.alphabet).encode(), np.uint8).copy()).cuda()
           for s in trip]
    want = oracle.align(*trip, sc.sub, sc.gap)
    for _ in range(2):
        out = torch.full((1,), -7, dtype=torch.int32, device="cuda")
        st = B.trioseq_align_noalloc(sc.alphabet, sc.sub, sc.gap, dev[0].data_ptr(), shape[0],
                                     dev[1].data_ptr(), shape[1], dev[2].data_ptr(), shape[2],
                                     out.data_ptr(), torch.cuda.current_stream())
        assert st == B.OK, B.trioseq_strerror(st)
        assert int(out.item()) == want
