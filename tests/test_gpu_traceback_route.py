"""The fused traceback explains every step of every path itself: the only pairs
that the int32 kernel traces are those that left the 16-bit range.  (A step that
nothing explained would send its pair there too, instead of a guessed path.)"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W
from test_gpu_band_edge import SCORINGS as EDGE, _pairs as _edge_pairs
from test_gpu_lazy import SCORINGS, _gap_pairs, _pairs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [5, 33, 100, 127, 200, 255, 500, 511, 639, 767])
def test_only_overflowing_pairs_are_traced_on_int32_lanes(w):
    batches = [make(w, W.replace(s, w=w), w, n=60) for s in SCORINGS.values() for make in (_gap_pairs, _pairs)]
    batches += [_edge_pairs(w, s) for s in EDGE]
    with A.Context(0) as ctx:
        for batch in batches:
            res, _, _ = ctx.align_cigar(A.pack_batch(batch), batch.scoring)
            end = np.where(res["reach_end"] == 1, res["mqe_t"], res["te"])
            info = ctx.last_traceback_info()
            assert info["pairs32"] == int(((res["lane16"] == 0) & (end >= 0)).sum()), (batch.scoring, info)
            assert info["fused"] == info["pairs16"] == batch.n_pairs
