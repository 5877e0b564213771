"""A peak just past the end of the table's head: the pair crosses the head's end,
goes back to a checkpoint before it, comes to the head's end again and there may
find that a rebase is due.  It must cross again as if for the first time; the
masked steps of the first crossing's range raised the maximum behind the blocks'
back, and the extension lost it.  Every field against the oracle (integers:
equality), over bands and rebase intervals that put the two together."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu

SCORINGS = [(40, 90, 60, 30, 200, 20), (250, 250, 0, 100, 0, 100), (100, 250, 20, 60, 20, 60),
            (200, 255, 100, 20, 240, 10), (255, 255, 0, 40, 0, 40), (60, 120, 0, 120, 0, 120),
            (30, 60, 30, 30, 100, 20)]


def _batch(si, w):
    """Sequences that part somewhere in the head, and a long pair for wide frames."""
    rng = np.random.default_rng(si * 1000 + w)
    qs, ts = [], []
    for _ in range(60):
        n = w + int(rng.integers(-3, 40))
        k = min(int(rng.integers(4, max(6, w))), n - 1) // 2
        x = rng.integers(0, 4, n, dtype=np.uint8)
        y = x.copy()
        y[k:] = np.where(rng.random(n - k) < rng.choice([0.3, 0.6, 0.9]), rng.integers(0, 4, n - k), y[k:])
        qs.append(x)
        ts.append(y)
    qs.append(rng.integers(0, 4, 600, dtype=np.uint8))
    ts.append(qs[-1].copy())
    return W.from_pairs(qs, ts, W.Scoring(*SCORINGS[si], w, -1 if w % 2 else 100000, 0))


@pytest.mark.parametrize("si", range(len(SCORINGS)))
def test_peak_past_the_heads_end(si):
    with A.Context(0) as ctx:
        for w in range(12, 100):
            batch = _batch(si, w)
            ref = O.align_batch(batch)
            got = A.agatha_align_batch(ctx, batch)
            bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
            assert bad.size == 0, (w, bad[:5])
            res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
            bad = A.results_equal(res, ref, O.COMPARE_FIELDS)
            assert bad.size == 0, ("cigar", w, bad[:5])
            want, _ = O.traceback_batch(batch, ref)
            assert all(np.array_equal(cig[off[i]:off[i + 1]], want[i]) for i in range(batch.n_pairs)), w
