"""The traceback's memory under a budget: its tables take what is left of it, and the
kept states of the fused form ask for what they take, not for a direction byte per
band slot and anti-diagonal."""
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


def _states(batch, C=16):
    n = batch.q_len.astype(np.int64) + batch.t_len - 1
    return (n // 32 + 1) * (384 * C + 16)


@pytest.mark.parametrize("lengths,waves", [([40000], 1), ([9000] * 12, 1), ([9000] * 12, 3)])
def test_a_budget_for_the_states_is_enough(lengths, waves):
    batch = _batch(lengths)
    states = _states(batch)
    rows = (batch.q_len.astype(np.int64) + batch.t_len - 1) * 512
    # besides the tables: results, sequences, runs and lists
    rest = (1 << 20) + 10 * int((batch.q_len.astype(np.int64) + batch.t_len).sum())
    room = int(states.sum()) if waves == 1 else int(states.max()) * -(-len(lengths) // waves)
    assert waves > 1 or room + rest < rows.sum()
    ref = O.align_batch(batch)
    want, _ = O.traceback_batch(batch, ref)
    with A.Context(0, mem_budget_bytes=room + rest) as ctx:
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
        info = ctx.last_traceback_info()
    assert info["waves"] <= waves and info["fused"] == batch.n_pairs, info
    assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0
    assert all(np.array_equal(cig[off[i]:off[i + 1]], want[i]) for i in range(batch.n_pairs))


@pytest.mark.parametrize("w", [100, 200, 500, 750])
def test_every_length_around_a_state(w):
    """Pairs whose last anti-diagonals lie around the first states kept."""
    lengths = list(range(1, 70)) + [4 * w]
    batch = _batch(lengths, w)
    ref = O.align_batch(batch)
    want, _ = O.traceback_batch(batch, ref)
    with A.Context(0) as ctx:
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
    assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0
    assert all(np.array_equal(cig[off[i]:off[i + 1]], want[i]) for i in range(batch.n_pairs))
