"""Steep scorings on lazy blocks: bands whose head the masked step would have to
run if cells off the table were asked to keep a bound from below, and tables
that the band covers.  Results and CIGARs against the oracle (all integers:
equality), and times against a mild scoring on the same pairs: the steps are
the same, so the times are."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W
from test_gpu_lazy import _gap_pairs, _pairs

pytestmark = pytest.mark.gpu

SCORINGS = {
    "asm5": W.Scoring(a=1, b=19, q=39, e=3, q2=81, e2=1, zdrop=-1),
    "b60": W.Scoring(a=1, b=60, q=10, e=20, q2=10, e2=20, zdrop=-1),
    "b250": W.Scoring(a=3, b=250, q=30, e=5, q2=60, e2=2, zdrop=-1),
    "head_too_steep": W.Scoring(a=64, b=64, q=1, e=63, q2=1, e2=63, zdrop=-1),
    "one_piece_b255": W.Scoring(a=255, b=255, q=0, e=40, q2=0, e2=40, zdrop=-1),
}


@pytest.fixture(scope="module")
def ctx():
    with A.Context(0, timing=True) as c:
        yield c


def _tables(w, scoring, seed):
    """Tables the band covers: up to its width, at the frame's and just longer."""
    rng = np.random.default_rng(seed)
    qs, ts = [], []
    for n in (1, 2, 9, 60, 100, 127, 128, 200, 254, 255, 256, 300, 400, w - 1, w, w + 1, w + 7, 510, 511, 512, 766, 767):
        for em in (W.ErrorModel(0.01, 0.01, 0.01), W.ErrorModel(0.15, 0.05, 0.05), W.ErrorModel(0.75, 0.0, 0.0)):
            q = rng.integers(0, 4, n, dtype=np.uint8)
            t, _ = W._mutate_chunk(rng, q, np.array([n], np.int32), em)
            qs.append(q)
            ts.append(t if len(t) else q)
    return W.from_pairs(qs, ts, W.replace(scoring, w=w))


@pytest.mark.parametrize("w", [100, 127, 255, 400, 500, 511, 600, 638, 750, 767])
@pytest.mark.parametrize("name", sorted(SCORINGS))
def test_results(ctx, name, w):
    s = W.replace(SCORINGS[name], w=w)
    for batch in (_tables(w, s, w), _pairs(w, s, seed=w, n=40), _gap_pairs(w, s, w, n=24)):
        ref = O.align_batch(batch)
        for flags in (0, A.AGATHA_REGS_HIGH, A.AGATHA_EDGE_PATH_ONLY):
            got = A.agatha_align_batch(ctx, batch, flags=flags)
            bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
            assert bad.size == 0, f"flags {flags:#x}: pairs {bad[:5]}"
        want, _ = O.traceback_batch(batch, ref)
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
        assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0
        bad = [i for i in range(batch.n_pairs) if not np.array_equal(cig[off[i]:off[i + 1]], want[i])]
        assert not bad, f"CIGARs of pairs {bad[:5]}"


@pytest.mark.parametrize("w,length", [(500, 300), (500, 600), (750, 600), (750, 1500)])
def test_time_as_of_a_mild_scoring(ctx, w, length):
    """The masked head took 2.5 to 4 times the mild scoring's time where the band
    covers the table and 1.8 to 2.4 where it does not (CIGARs: 2 to 4)."""
    rng = np.random.default_rng(w)
    qs, ts = [], []
    for _ in range(3000):
        q = rng.integers(0, 4, length, dtype=np.uint8)
        t, _ = W._mutate_chunk(rng, q, np.array([length], np.int32), W.ErrorModel(0.002, 0.0, 0.0))
        qs.append(q)
        ts.append(t)
    score, cigar = {}, {}
    for name, s in (("mild", W.replace(W.ONT_SCORING, w=w, zdrop=-1)), ("steep", W.replace(SCORINGS["asm5"], w=w))):
        pb = A.pack_batch(W.from_pairs(qs, ts, s))
        a, b = [], []
        for _ in range(7):
            ctx.align_host(pb, s)
            a.append(ctx.last_kernel_ms())
            ctx.align_cigar(pb, s)
            b.append(ctx.last_traceback_ms())
        score[name], cigar[name] = sorted(a)[2], sorted(b)[2]
    assert score["steep"] < 1.5 * score["mild"], score
    assert cigar["steep"] < 1.5 * cigar["mild"], cigar
