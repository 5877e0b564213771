"""The autotuner on 24-slot bands, where lazy blocks have one register budget: it
never chooses between a kernel and itself (noise would decide), and a file that
names the second budget there still gives a plan."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _batch(zdrop):
    rng = np.random.default_rng(1)
    qs, ts = [], []
    for n in [300] * 20 + [900] * 6 + [3000] * 2 + [9000]:
        q = rng.integers(0, 4, n, dtype=np.uint8)
        t, _ = W._mutate_chunk(rng, q, np.array([n], np.int32), W.ErrorModel(0.05, 0.03, 0.03))
        qs.append(q)
        ts.append(t)
    return W.from_pairs(qs, ts, W.replace(W.ONT_SCORING, w=600, zdrop=zdrop))


def test_one_budget_is_not_tuned():
    with A.Context(0, autotune=True) as ctx:
        for zdrop in range(400, 460):                # a key of its own each
            batch = _batch(zdrop)
            A.agatha_align_batch(ctx, batch)
            assert 1 not in ctx.tune_variants(batch.scoring)[:4], zdrop


@pytest.mark.parametrize("plan", ["1 1 1 1 0", "3 1 0 1 1", "1 2 1 0 1"])
def test_a_file_naming_the_second_budget(tmp_path, plan):
    import torch
    batch = _batch(400)
    s = batch.scoring
    prop = torch.cuda.get_device_properties(0)
    path = tmp_path / "tune.txt"
    path.write_text(f"sm{prop.multi_processor_count}_cc{prop.major}{prop.minor}_a{s.a}_b{s.b}_q{s.q}_e{s.e}"
                    f"_q2{s.q2}_e2{s.e2}_w{s.w}_z{s.zdrop}_c24 {plan}\n")
    with A.Context(0, autotune=True, tune_cache_path=str(path)) as ctx:
        got = A.agatha_align_batch(ctx, batch)
        assert ctx.tune_variants(s) == [int(x) for x in plan.split()]
    assert A.results_equal(got, O.align_batch(batch), O.COMPARE_FIELDS).size == 0
