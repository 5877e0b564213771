"""The kernels that test every anti-diagonal, which scorings whose Z-drop
threshold leaves lazy blocks no room run on: every field of every pair and
every CIGAR against the oracle on both sides of the line between the two (all
integers: equality), and that such a threshold costs no more than that step
does."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W
from test_gpu_lazy import _gap_pairs, _pairs

pytestmark = pytest.mark.gpu

SCORINGS = {
    "ont": W.ONT_SCORING,
    "bwa": W.BWA_SCORING,
    "asm5": W.Scoring(a=1, b=19, q=39, e=3, q2=81, e2=1),
    "short": W.Scoring(a=2, b=8, q=12, e=2, q2=24, e2=1),
    "second_cheaper": W.Scoring(a=2, b=4, q=4, e=6, q2=5, e2=1, end_bonus=3),
    "steep": W.Scoring(a=200, b=250, q=0, e=215, q2=0, e2=215),      # too steep for kept states
}


def line(s):
    """The least threshold at which the lazy blocks run."""
    if s.q2 <= s.q or s.e2 >= s.e:
        q, e = s.q, s.e
    elif s.q + s.e > s.q2 + s.e2:
        q, e = s.q2, s.e2
    else:
        q, e = s.q, s.e
    c = max(s.b, 2 * e)
    return 2 * q + e + 5 * c + max(4 * s.a, q + e)


@pytest.fixture(scope="module")
def ctx():
    with A.Context(0, timing=True) as c:
        yield c


def _cigars(ctx, batch, ref, flags=0):
    res, off, cig = ctx.align_cigar(A.pack_batch(batch), batch.scoring, flags=flags)
    assert A.results_equal(res, ref, O.COMPARE_FIELDS).size == 0, f"flags {flags:#x}"
    want, _ = O.traceback_batch(batch, ref)
    bad = [i for i in range(batch.n_pairs) if not np.array_equal(cig[off[i]:off[i + 1]], want[i])]
    assert not bad, f"flags {flags:#x}: CIGARs of pairs {bad[:5]}"


@pytest.mark.parametrize("w", [5, 8, 100, 127, 128, 255, 256, 500, 511, 512, 630, 639, 750, 767, 768, 1000, 1023])
@pytest.mark.parametrize("name", sorted(SCORINGS))
def test_both_sides_of_the_line(ctx, name, w):
    s = SCORINGS[name]
    for z in (0, line(s) // 2, line(s) - 1, line(s)):
        for make in (_pairs, _gap_pairs):
            batch = make(w, W.replace(s, w=w, zdrop=z), seed=w + z, n=40)
            ref = O.align_batch(batch)
            for flags in (0, A.AGATHA_REGS_HIGH, A.AGATHA_FORCE32, A.AGATHA_ONE_FRAME, A.AGATHA_NO_SORT):
                got = A.agatha_align_batch(ctx, batch, flags=flags)
                bad = A.results_equal(got, ref, O.COMPARE_FIELDS)
                assert bad.size == 0, f"z {z} flags {flags:#x}: pairs {bad[:5]}"
            _cigars(ctx, batch, ref)


@pytest.mark.parametrize("w", [100, 500, 1000])
def test_allocation_free_below_the_line(w):
    torch = pytest.importorskip("torch")
    batch = _pairs(w, W.replace(W.ONT_SCORING, w=w, zdrop=30), seed=w)
    pb = A.pack_batch(batch)
    dev = {k: torch.from_numpy(getattr(pb, k)).cuda() for k in
           ("q_packed", "t_packed", "q_off", "t_off", "q_len", "t_len")}
    out = torch.zeros(pb.n_pairs * 48, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    A.agatha_align_batch_noalloc(out=out, scoring=batch.scoring, **dev)
    got = out.cpu().numpy().view(A.RESULT_DTYPE)
    assert A.results_equal(got, O.align_batch(batch), O.COMPARE_FIELDS).size == 0


def test_tuned_and_split_below_the_line(tmp_path):
    """Both register budgets and int32 lanes, per length class and alone."""
    import torch
    s = W.replace(W.ONT_SCORING, w=500, zdrop=30)
    batch = _pairs(500, s, seed=3, n=200)
    ref = O.align_batch(batch)
    prop = torch.cuda.get_device_properties(0)
    key = (f"sm{prop.multi_processor_count}_cc{prop.major}{prop.minor}_a{s.a}_b{s.b}_q{s.q}_e{s.e}"
           f"_q2{s.q2}_e2{s.e2}_w{s.w}_z{s.zdrop}_c16")
    for plan in ("1 1 1 1 0", "2 2 2 2 0", "0 1 2 0 1"):
        path = tmp_path / "tune.txt"
        path.write_text(f"{key} {plan}\n")
        with A.Context(0, autotune=True, tune_cache_path=str(path)) as c:
            assert A.results_equal(A.agatha_align_batch(c, batch), ref, O.COMPARE_FIELDS).size == 0
    with A.Context(0, autotune=True) as c:
        assert A.results_equal(A.agatha_align_batch(c, batch), ref, O.COMPARE_FIELDS).size == 0


def _accurate(n, length, scoring):
    rng = np.random.default_rng(7)
    qs, ts = [], []
    for _ in range(n):
        q = rng.integers(0, 4, length, dtype=np.uint8)
        t, _ = W._mutate_chunk(rng, q, np.array([length], np.int32), W.ErrorModel(0.002, 0.0, 0.0))
        qs.append(q)
        ts.append(t)
    return W.from_pairs(qs, ts, scoring)


@pytest.mark.parametrize("w,length,flags,limit", [(100, 600, 0, 3.0), (500, 2000, 0, 3.0),
                                                  (500, 1500, A.AGATHA_FORCE32, 3.3)])
def test_a_low_threshold_costs_no_more_than_its_step(ctx, w, length, flags, limit):
    """The step that tests every anti-diagonal takes 1.5 to 2.1 times the lazy
    step's time on these (2.3 on int32 lanes), the lazy drive's masked step 4.5
    to 5.5 times (4.3): the limits lie between."""
    n = 6000 if length == 600 else 1500
    ms = {}
    for z in (30, -1):
        pb = A.pack_batch(_accurate(n, length, W.replace(W.ONT_SCORING, w=w, zdrop=z)))
        s = W.replace(W.ONT_SCORING, w=w, zdrop=z)
        t = []
        for _ in range(7):
            ctx.align_host(pb, s, flags=flags)
            t.append(ctx.last_kernel_ms())
        ms[z] = sorted(t)[2]
    assert ms[30] < limit * ms[-1], ms


def test_a_low_threshold_costs_no_more_for_cigars(ctx):
    """As above for the fused traceback: 1.5 to 2 against 3.3."""
    ms = {}
    for z in (30, -1):
        s = W.replace(W.ONT_SCORING, w=100, zdrop=z)
        pb = A.pack_batch(_accurate(3000, 600, s))
        t = []
        for _ in range(7):
            ctx.align_cigar(pb, s)
            t.append(ctx.last_traceback_ms())
        ms[z] = sorted(t)[2]
    assert ms[30] < 2.6 * ms[-1], ms


@pytest.mark.parametrize("w,n", [(600, 1), (600, 700), (600, 800), (1000, 1), (1000, 900), (1000, 950)])
def test_three_warps_below_the_line(ctx, w, n):
    """int32 lanes on bands of more than 511: three warps per pair up to one wave
    of them (two for the widest), one warp beyond."""
    rng = np.random.default_rng(n)
    qs = [rng.integers(0, 4, 640 if i else 1300, dtype=np.uint8) for i in range(n)]
    ts = [W._mutate_chunk(rng, q, np.array([len(q)], np.int32), W.ErrorModel(0.02, 0.01, 0.01))[0] for q in qs]
    batch = W.from_pairs(qs, ts, W.replace(W.ONT_SCORING, w=w, zdrop=30))
    got = A.agatha_align_batch(ctx, batch, flags=A.AGATHA_FORCE32)
    assert A.results_equal(got, O.align_batch(batch), O.COMPARE_FIELDS).size == 0


def test_a_lone_wide_pair_keeps_three_warps(ctx):
    """4.5 times the lazy time on the masked step of three warps, 9.5 on one warp."""
    ms = {}
    for z in (30, -1):
        s = W.replace(W.ONT_SCORING, w=1000, zdrop=z)
        pb = A.pack_batch(_accurate(1, 3000, s))
        t = []
        for _ in range(7):
            ctx.align_host(pb, s)
            t.append(ctx.last_kernel_ms())
        ms[z] = sorted(t)[2]
    assert ms[30] < 6.5 * ms[-1], ms
