"""The lazy blocks of the 16-bit and int32 kernels against the oracle, every field of every
pair, where the blocks can go wrong: bands whose edge falls in each register
of a lane (and in the frame's last slot), tables shorter than the band or
just longer, tables whose corner leaves the band, ends of every parity,
divergent tails (the Z-drop bound), long indels (a peak passed and taken
back), and scorings at the edges of the drift (one piece, the second piece
always the cheaper, an extension dearer than a match, steep enough for a
rebase in every block).  Every output is an integer: equality."""
import numpy as np
import pytest

from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu

TWO = W.ONT_SCORING
ONE = W.BWA_SCORING
SCORINGS = {
    "two": TWO,
    "one": ONE,
    "second_cheaper": W.Scoring(a=2, b=4, q=4, e=6, q2=5, e2=1, zdrop=200, end_bonus=3),
    "dear_extension": W.Scoring(a=1, b=1, q=0, e=1, q2=0, e2=1, zdrop=60),
    "steep": W.Scoring(a=40, b=90, q=60, e=30, q2=200, e2=20, zdrop=3000),
    "no_zdrop": W.Scoring(a=2, b=4, q=4, e=2, q2=24, e2=1, zdrop=-1),
    "free_mismatch": W.Scoring(a=1, b=0, q=2, e=1, q2=2, e2=1, zdrop=30),
}


def _pairs(w, scoring, seed, n=72):
    rng = np.random.default_rng(seed)
    qs, ts = [], []
    lens = [1, 2, 3, 7, 33, w // 2, w - 3, w - 1, w, w + 1, w + 2, w + 3, w + 5, w + 9, w + 40, 2 * w, 2 * w + 1,
            3 * w + 11, 5 * w + 300]
    for i in range(n):
        ql = max(1, lens[i % len(lens)] + int(rng.integers(0, 3)))
        q = rng.integers(0, 4, ql, dtype=np.uint8)
        em = W.ErrorModel(0.06, 0.03, 0.03, tail_frac=0.3 if i % 3 else 0.0)
        t, _ = W._mutate_chunk(rng, q, np.array([ql], np.int32), em)
        if i % 5 == 1 and len(t) > 80:              # a long gap: the maximum falls and recovers
            k = int(rng.integers(2, max(4, min(60, w))))
            at = int(rng.integers(10, len(t) - 70))
            t = np.concatenate([t[:at], t[at + k:]])
        if i % 7 == 2:                               # the corner off the band, or nearly
            t = t[:max(1, len(t) - w + int(rng.integers(-2, 3)))]
        if i % 11 == 3:
            t = np.concatenate([t, rng.integers(0, 4, w + int(rng.integers(-2, 3)), dtype=np.uint8)])
        qs.append(q)
        ts.append(t if len(t) else np.zeros(1, np.uint8))
    return W.from_pairs(qs, ts, scoring)


@pytest.fixture(scope="module")
def ctx():
    with A.Context(0) as c:
        yield c


BANDS = [5, 8, 9, 100, 101, 102, 103, 126, 127, 128, 131, 132, 133, 134, 255, 256] + list(range(493, 513)) + \
        [630, 638, 639, 640, 744, 751, 755, 758, 759, 760, 766, 767]


@pytest.mark.parametrize("w", BANDS)
def test_bands(ctx, w):
    from oracle import oracle as O
    scoring = ONE if w % 2 else TWO
    batch = _pairs(w, W.replace(scoring, w=w), seed=w)
    ref = O.align_batch(batch)
    for flags in (0, A.AGATHA_REGS_HIGH):
        got = A.agatha_align_batch(ctx, batch, flags=flags)
        bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
        assert bad.size == 0, f"pairs {bad[:5]}"
        assert got["lane16"].all()


@pytest.mark.parametrize("w", [5, 8, 100, 127, 128, 200, 255, 500, 511, 512, 750, 767, 768] +
                         list(range(990, 1024)))
def test_bands_int32(ctx, w):
    from oracle import oracle as O
    batch = _pairs(w, W.replace(ONE if w % 2 else TWO, w=w), seed=5000 + w)
    ref = O.align_batch(batch)
    got = A.agatha_align_batch(ctx, batch, flags=A.AGATHA_FORCE32)
    bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
    assert bad.size == 0, f"pairs {bad[:5]}"
    assert not got["lane16"].any()


@pytest.mark.parametrize("w", [100, 200, 500, 750])
@pytest.mark.parametrize("name", sorted(SCORINGS))
def test_scorings(ctx, name, w):
    from oracle import oracle as O
    batch = _pairs(w, W.replace(SCORINGS[name], w=w), seed=1000 + w)
    ref = O.align_batch(batch)
    for flags in (0, A.AGATHA_FORCE32):
        got = A.agatha_align_batch(ctx, batch, flags=flags)
        bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
        assert bad.size == 0, f"flags {flags}: pairs {bad[:5]}"


@pytest.mark.parametrize("w", [100, 500, 1000])
def test_int32_large_scores(ctx, w):
    """Scores near the int32 headroom the library admits (2^28 for the
    pair's anti-diagonals), far beyond 16-bit lanes."""
    from oracle import oracle as O
    batch = _pairs(w, W.Scoring(a=4000, b=7000, q=1500, e=1200, q2=7000, e2=600, w=w, zdrop=200000), seed=77 + w)
    ref = O.align_batch(batch)
    got = A.agatha_align_batch(ctx, batch)
    bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
    assert bad.size == 0, f"pairs {bad[:5]}"


def _gap_pairs(w, scoring, seed, n=48):
    """Pairs whose paths hold gaps of up to several segments of the
    traceback's recomputation, in either sequence, and leading gaps."""
    rng = np.random.default_rng(seed)
    qs, ts = [], []
    for i in range(n):
        x = rng.integers(0, 4, int(rng.integers(60, 900)), dtype=np.uint8)
        y, _ = W._mutate_chunk(rng, x, np.array([len(x)], np.int32), W.ErrorModel(0.03, 0.02, 0.02))
        for _ in range(2):
            k = int(rng.integers(1, max(2, min(200, w))))
            at = int(rng.integers(0, max(1, len(y) - k))) if i % 4 else 0
            y = np.concatenate([y[:at], y[at + k:]])
        if not len(y):
            y = x[:1]
        if i % 3 == 0:                          # repeats: ties between gap places
            y = np.concatenate([y, np.tile(x[:7], 9)])
        qs.append(x if i % 2 else y)
        ts.append(y if i % 2 else x)
    return W.from_pairs(qs, ts, scoring)


@pytest.mark.parametrize("w", [5, 8, 33, 100, 127, 128, 200, 255, 500, 511, 630, 750, 767])
@pytest.mark.parametrize("name", sorted(SCORINGS))
def test_cigars(ctx, name, w):
    from oracle import oracle as O
    for make, seed in ((_gap_pairs, 31), (_pairs, 32)):
        batch = make(w, W.replace(SCORINGS[name], w=w), seed + w, n=40)
        ref = O.align_batch(batch)
        want, _ = O.traceback_batch(batch, ref)
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
        bad = A.results_equal(res, ref, O.COMPARE_FIELDS)
        assert bad.size == 0, f"results of pairs {bad[:5]}"
        for i in range(batch.n_pairs):
            got = cig[off[i]:off[i + 1]]
            assert np.array_equal(got, want[i]), (i, A.cigar_string(got), A.cigar_string(want[i]))


@pytest.mark.parametrize("w", [4, 5, 8, 13, 33, 100, 101, 102, 126, 127, 128, 200, 255, 256, 300, 500, 510, 511])
@pytest.mark.parametrize("name", ["one", "two", "second_cheaper", "dear_extension", "no_zdrop", "free_mismatch"])
def test_local(ctx, name, w):
    """The local extension's row blocks: initial scores that die before, at and
    after the band's corner (the last take the per-cell step), rows that end
    with the band and with the table, and scores too large for the row keys."""
    from oracle import oracle as O
    rng = np.random.default_rng(900 + w)
    for make in (_pairs, _gap_pairs):
        batch = make(w, W.replace(SCORINGS[name], w=w), 77 + w, n=60)
        edge = [1, 2, 7, 20, 40, 60, w, w + 7, 2 * w + 9, 1000, (1 << 20) - 3, 1 << 24]
        h0 = rng.choice(edge, batch.n_pairs).astype(np.int32)
        ref = O.align_batch(batch, h0=h0)
        got = ctx.align_local(A.pack_batch(batch), batch.scoring, h0)
        bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
        assert bad.size == 0, (bad[:5], h0[bad[:5]], got[bad[:2]], ref[bad[:2]])


@pytest.mark.parametrize("n", [1, 3, 151, 153, 607, 609, 1217, 1825, 2500, 4096, 4097])
@pytest.mark.parametrize("w", [100, 200, 500, 750, 1000])
def test_tiers(ctx, n, w):
    """Batches that just fill a tier of the SMs' warps or not quite, with a few
    pairs that bound the launch (whose later tiers stay away) or none, sorted
    and unsorted, prepared in one launch (up to 4,096) and in three: every pair
    is aligned once."""
    from oracle import oracle as O
    for long_ones in (0, min(n, 9)):
        rng = np.random.default_rng(n + w + long_ones)
        qs, ts = [], []
        for i in range(n):
            ql = int(rng.integers(30, 60)) if i >= long_ones else int(rng.integers(900, 1500))
            q = rng.integers(0, 4, ql, dtype=np.uint8)
            t, _ = W._mutate_chunk(rng, q, np.array([ql], np.int32), W.ErrorModel(0.05, 0.03, 0.03))
            qs.append(q)
            ts.append(t if len(t) else q)
        batch = W.from_pairs(qs, ts, W.replace(TWO, w=w))
        ref = O.align_batch(batch)
        for flags in (0, A.AGATHA_FORCE32, A.AGATHA_NO_SORT):
            got = A.agatha_align_batch(ctx, batch, flags=flags)
            bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
            assert bad.size == 0, (flags, bad[:5])
        if w < 768:
            res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
            assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0
            want, _ = O.traceback_batch(batch, ref)
            assert all(np.array_equal(cig[off[i]:off[i + 1]], want[i]) for i in range(n))


@pytest.mark.parametrize("n", [1, 153, 609, 2500, 4097])
@pytest.mark.parametrize("w", [100, 200, 500])
def test_local_tiers(ctx, n, w):
    """The local extension's queue over the tiers of the SMs' warps, some pairs
    bounding the launch and some for the per-cell step."""
    from oracle import oracle as O
    rng = np.random.default_rng(5 * n + w)
    qs, ts = [], []
    for i in range(n):
        q = rng.integers(0, 4, int(rng.integers(30, 60) if i >= 9 else rng.integers(700, 1100)), dtype=np.uint8)
        t, _ = W._mutate_chunk(rng, q, np.array([len(q)], np.int32), W.ErrorModel(0.05, 0.03, 0.03))
        qs.append(q)
        ts.append(t if len(t) else q)
    batch = W.from_pairs(qs, ts, W.replace(ONE, w=w))
    h0 = rng.integers(19, 61, n).astype(np.int32)
    h0[::17] = 1 << 24
    ref = O.align_batch(batch, h0=h0)
    for flags in (0, A.AGATHA_NO_SORT):
        got = ctx.align_local(A.pack_batch(batch), batch.scoring, h0, flags=flags)
        assert A.results_equal(got, ref, O.COMPARE_FIELDS).size == 0
