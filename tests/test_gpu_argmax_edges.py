"""Rows that start at every 4-byte alignment: the row maxima are read in 16-byte
words from the first 16-byte boundary of a slice on, and the elements before it
and after the last whole word one by one.  Indices are compared exactly."""
import numpy as np
import pytest

from tests.test_gpu_commit import check_accept

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,W", [(1, 8), (9, 16)])  # one kernel, two kernels
@pytest.mark.parametrize("V", [1, 2, 3, 5, 6, 7, 9, 33, 4097, 4098, 4099, 50257])
def test_maximum_at_the_ends(B, W, V):
    """The maximum in each of the first and last five columns, then equal maxima at
    both ends (the first wins), over rows of all alignments."""
    ends = sorted(set(c for c in [*range(5), *range(V - 5, V)] if 0 <= c < V))
    rng = np.random.default_rng(V)
    logits = rng.standard_normal((B, W, V), dtype=np.float32)
    first = np.zeros((B, W), dtype=np.int64)
    for n in range(B * W):
        b, w = divmod(n, W)
        c = ends[n % len(ends)]
        logits[b, w, c] = 9.0
        if n % 3 == 0:
            logits[b, w, V - 1] = 9.0
        first[b, w] = c
    _, tid, _ = check_accept(logits, np.zeros((B, W), dtype=np.int32))
    assert np.array_equal(tid, first)
