"""A peak within a rebase interval of the end: the pair goes back to a
checkpoint from which the next rebase is only a few anti-diagonals away, and must
rebase there from the checkpoint's own maximum.  With the maximum of the place it
came back from, pairs whose scores had risen since failed the rebase's check and
went to int32 lanes.  The scorings' steps are near the largest that 16-bit lanes
take, and the bands' spread of scores near what they hold.  Results and CIGARs
against the oracle (equality); the listed pairs stay on 16-bit lanes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _batch(seed, w, e, a, b, n=2000):
    """Equal sequences, one a few bases off the band's middle, with a diverging end."""
    rng = np.random.default_rng(seed)
    qs, ts = [], []
    for i in range(n):
        length = int(rng.integers(2 * w, 2 * w + 260))
        d = int(rng.integers(0, 8))
        k = int(rng.integers(0, 60))
        x = rng.integers(0, 4, length, dtype=np.uint8)
        t = np.concatenate([rng.integers(0, 4, d, dtype=np.uint8), x])
        q = x.copy()
        if k:
            q[-k:] = np.where(rng.random(k) < rng.choice([0.2, 0.5, 0.9]), rng.integers(0, 4, k), q[-k:])
        if i % 3 == 0:
            t = np.concatenate([t, rng.integers(0, 4, int(rng.integers(0, 40)), dtype=np.uint8)])
        if i % 2:
            t, q = q, t
        qs.append(q)
        ts.append(t)
    return W.from_pairs(qs, ts, W.Scoring(a, b, 0, e, 0, e, w, -1, 0))


# band, extension, match, mismatch; pairs to stay on 16-bit lanes in the score path and with CIGARs
CASES = [
    (111, 250, 100, 250, [128, 1280], []),
    (110, 250, 100, 250, [], [27, 310, 1537, 1574, 1609]),
    (109, 250, 100, 250, [493, 1349], [458, 462, 493, 1366, 1585]),
    (107, 250, 100, 250, [137, 1345], [137, 163, 272, 401, 457, 494, 820, 860, 955, 1458, 1627, 1661]),
    (130, 150, 200, 255, [], [1719]),
    (596, 40, 30, 100, [], []),
]


@pytest.mark.parametrize("w,e,a,b,score16,cigar16", CASES)
def test_peak_before_a_rebase(w, e, a, b, score16, cigar16):
    batch = _batch(w, w, e, a, b, n=2000 if w < 500 else 300)
    ref = O.align_batch(batch)
    with A.Context(0) as ctx:
        got = A.agatha_align_batch(ctx, batch)
        assert A.results_equal(got, ref, O.COMPARE_FIELDS).size == 0
        assert got["lane16"][score16].all(), [i for i in score16 if not got["lane16"][i]]
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
        assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0
        assert res["lane16"][cigar16].all(), [i for i in cigar16 if not res["lane16"][i]]
        idx = np.unique(np.concatenate([np.asarray(cigar16, np.int64), np.arange(0, batch.n_pairs, 7)]))
        want, _ = O.traceback_batch(batch, {int(i): ref[i] for i in idx}, idx)
        for k, i in enumerate(idx):
            assert np.array_equal(cig[off[i]:off[i + 1]], want[k]), i
