"""The traceback's memory under a budget."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _batch(lengths, w=500):
    rng = np.random.default_rng(3)
    qs, ts = [], []
    for n in lengths:
        q = rng.integers(0, 4, n, dtype=np.uint8)
        t, _ = W._mutate_chunk(rng, q, np.array([n], np.int32), W.ErrorModel(0.05, 0.03, 0.03))
        qs.append(q)
        ts.append(t)
    return W.from_pairs(qs, ts, W.replace(W.ONT_SCORING, w=w))


@pytest.mark.parametrize("flags", [0, A.AGATHA_TB_TWO_PASS, A.AGATHA_FORCE32])
@pytest.mark.parametrize("odd", [0, 1, 100, 255])
def test_waves_under_any_budget(flags, odd):
    """The tables take what a budget leaves, whether or not that is a whole number
    of the allocator's granules."""
    batch = _batch([6000] * 24)
    with A.Context(0) as big:
        r1, o1, c1 = big.align_cigar(A.pack_batch(batch), batch.scoring, flags=flags)
    with A.Context(0, mem_budget_bytes=(28 << 20) + odd) as small:
        r2, o2, c2 = small.align_cigar(A.pack_batch(batch), batch.scoring, flags=flags)
        assert small.last_traceback_info()["waves"] > 1
    assert A.results_equal(r1, r2).size == 0
    assert np.array_equal(o1, o2) and np.array_equal(c1, c2)
