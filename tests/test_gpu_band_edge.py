"""Paths that only the virtual column (row) beyond the band could give, in
every kernel, against the oracle: the virtual cells (t, -1) and (-1, q) have no
band, but the table's cells next to them with t > w (q > w) are outside it, so
a gap out of such a virtual cell ends there and must not come back into the
band two or more anti-diagonals later.  Every output is an integer: equality."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu

# mismatches dearer than two gaps, so that a path through the corner of the band
# pays for each change of direction
SCORINGS = [W.Scoring(a=5, b=60, q=20, e=1, q2=20, e2=1, zdrop=-1, end_bonus=20000),
            W.Scoring(a=5, b=90, q=10, e=4, q2=30, e2=1, zdrop=4000),
            W.Scoring(a=5, b=19, q=39, e=3, q2=81, e2=1, zdrop=-1)]


def _pairs(w, scoring):
    rng = np.random.default_rng(w)
    qs, ts = [], []
    for k in range(0, 5):
        for n in (0, 1, 40, 400 if w > 127 else 90):
            x = rng.integers(0, 4, n, dtype=np.uint8)
            for gap in (w - 1, w, w + 1):       # the diagonal of x, around the band's edge
                long, short = np.zeros(k + gap, np.uint8), np.ones(max(k, 1), np.uint8)
                for m in (x, np.concatenate([x, rng.integers(0, 4, 9, dtype=np.uint8)])):
                    ts += [np.concatenate([long, x]), np.concatenate([short, m])]
                    qs += [np.concatenate([short, m]), np.concatenate([long, x])]
    for _ in range(40):                         # and unrelated sequences
        qs.append(rng.integers(0, 4, int(rng.integers(1, 3 * w + 9)), dtype=np.uint8))
        ts.append(rng.integers(0, 4, int(rng.integers(1, 3 * w + 9)), dtype=np.uint8))
    return W.from_pairs(qs, ts, W.replace(scoring, w=w))


@pytest.fixture(scope="module")
def ctx():
    with A.Context(0) as c:
        yield c


def _score_routes(w):
    routes = [0, A.AGATHA_REGS_HIGH, A.AGATHA_EDGE_PATH_ONLY, A.AGATHA_FORCE32, A.AGATHA_PLAIN,
              A.AGATHA_FORCE32 | A.AGATHA_EDGE_PATH_ONLY]
    if w <= 127:
        routes.append(A.AGATHA_HALF_WARP)
    if 256 <= w <= 767:
        routes += [A.AGATHA_WARPS2, A.AGATHA_WARPS4]
    return routes


@pytest.mark.parametrize("si", range(len(SCORINGS)))
@pytest.mark.parametrize("w", [5, 8, 9, 100, 127, 128, 255, 300, 511, 600, 767, 900])
def test_band_edge(ctx, w, si):
    batch = _pairs(w, SCORINGS[si])
    ref = O.align_batch(batch)
    for flags in _score_routes(w):
        got = A.agatha_align_batch(ctx, batch, flags=flags)
        bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
        assert bad.size == 0, f"flags {flags:#x}: {bad.size} pairs, first {bad[0]}"
    want, _ = O.traceback_batch(batch, ref)
    for flags in (0, A.AGATHA_TB_TWO_PASS, A.AGATHA_FORCE32):
        res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring, flags=flags)
        assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0, f"flags {flags:#x}"
        bad = [i for i in range(batch.n_pairs) if not np.array_equal(cig[off[i]:off[i + 1]], want[i])]
        assert not bad, (f"flags {flags:#x}: {len(bad)} CIGARs, first {bad[0]}: "
                         f"{A.cigar_string(cig[off[bad[0]]:off[bad[0] + 1]])[:80]}, "
                         f"want {A.cigar_string(want[bad[0]])[:80]}")
    if w <= 511:
        h0 = np.full(batch.n_pairs, 3 * w + 60, np.int32)
        got = ctx.align_local(A.pack_batch(batch), batch.scoring, h0)
        assert A.results_equal(got, O.align_batch(batch, h0=h0), O.COMPARE_FIELDS).size == 0


@pytest.mark.parametrize("w", [8, 200, 600, 900])
def test_band_edge_allocation_free(w):
    torch = pytest.importorskip("torch")
    for scoring in SCORINGS:
        batch = _pairs(w, scoring)
        pb = A.pack_batch(batch)
        dev = {k: torch.from_numpy(getattr(pb, k)).cuda() for k in
               ("q_packed", "t_packed", "q_off", "t_off", "q_len", "t_len")}
        out = torch.zeros(pb.n_pairs * 48, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        A.agatha_align_batch_noalloc(out=out, scoring=batch.scoring, **dev)
        got = out.cpu().numpy().view(A.RESULT_DTYPE)
        assert A.results_equal(got, O.align_batch(batch), O.COMPARE_FIELDS).size == 0
