"""Mask words to one byte per register, at the edges of words and of the vector width: against numpy.unpackbits."""
import numpy as np
import pytest

from paper_2506_17506_b200 import binding


@pytest.mark.parametrize("n,P", [(0, 8), (1, 1), (3, 31), (5, 32), (4, 33), (7, 63), (2, 64), (3, 65), (6, 256), (5, 1000)])
def test_expand_masks(n, P):
    W = (P + 31) // 32
    words = np.random.default_rng(P).integers(0, 2**32, (n, W), dtype=np.uint32)
    out = np.full((n, P), 7, dtype=np.uint8)
    assert binding._lib.vl_expand_masks(words.ctypes.data, n, P, out.ctypes.data) == 0
    want = np.unpackbits(words.view(np.uint8).reshape(n, W * 4), axis=1, bitorder="little")[:, :P]
    assert (out == want).all()
