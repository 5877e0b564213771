"""The local extension's row blocks over drifts that take the row keys past 32 bits:
dear extensions over thousands of anti-diagonals, against the oracle (equality)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scoring", [W.Scoring(20, 40, 100, 400, 100, 400, 100, 100000, 5),
                                     W.Scoring(20, 60, 100, 500, 900, 300, 100, -1, 0)])
def test_long_drift(scoring):
    rng = np.random.default_rng(5)
    qs, ts = [], []
    for n in (500, 2500, 2700, 4000, 6000, 9000):
        for rate in (0.005, 0.03):
            q = rng.integers(0, 4, n, dtype=np.uint8)
            t, _ = W._mutate_chunk(rng, q, np.array([n], np.int32), W.ErrorModel(rate, rate / 10, rate / 10))
            qs.append(q)
            ts.append(t)
    batch = W.from_pairs(qs, ts, scoring)
    # drift e2 (tlen + qlen) beyond 2^21, scores below the row keys' 2^20
    assert scoring.e2 * int((batch.t_len + batch.q_len).max()) > 1 << 22
    h0 = np.full(batch.n_pairs, 2000, np.int32)
    with A.Context(0) as ctx:
        got = ctx.align_local(A.pack_batch(batch), scoring, h0)
    assert A.results_equal(got, O.align_batch(batch, h0=h0), O.COMPARE_FIELDS).size == 0
