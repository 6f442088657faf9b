"""Marshalling of triplets in the binding (no GPU): one triplet takes a path of its own, and accepts
every sized collection that a batch is accepted in, with the same records."""
import collections
import ctypes

import numpy as np
import pytest

from paper_2605_28400_gb300 import binding as B

COLLECTIONS = {"list": list, "tuple": tuple, "deque": collections.deque, "set": set,
               "dict values": lambda t: dict(enumerate(t)).values(),
               "array": lambda t: np.array(t)}


def _records(triplets):
    arr, keep = B._triplet_array(triplets)
    ptr = ctypes.POINTER(ctypes.c_void_p)
    out = [tuple(ctypes.string_at(ctypes.cast(ctypes.byref(arr[i], B.Triplet.s.offset), ptr)[q],
                                  arr[i].len[q]) for q in range(3)) for i in range(len(triplets))]
    del keep
    return out


@pytest.mark.parametrize("kind", COLLECTIONS)
@pytest.mark.parametrize("n", [1, 2])
def test_every_collection(kind, n):
    trips = [("ACGT", "", "GG"), ("A", "CC", "TTTT")][:n]
    want = [tuple(x.encode() for x in t) for t in trips]
    assert sorted(_records(COLLECTIONS[kind](trips))) == sorted(want)


@pytest.mark.parametrize("parts", [(b"ACGT", b"", b"GG"), ("ACGT", b"", b"GG"),
                                   (np.frombuffer(b"ACGT", np.uint8), "", bytearray(b"GG"))])
def test_bytes_and_code_arrays(parts):
    for n in (1, 2):
        assert _records([parts] * n) == [(b"ACGT", b"", b"GG")] * n
