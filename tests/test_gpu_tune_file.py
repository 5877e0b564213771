"""The autotuner's file belongs to the build that measured it."""
import pytest

from paper_2403_06478_gb300 import agatha as A
from paper_2403_06478_gb300 import workload as W

pytestmark = pytest.mark.gpu


def _tuned(path, batch):
    with A.Context(0, autotune=True, tune_cache_path=str(path)) as ctx:
        A.agatha_align_batch(ctx, batch)
        return ctx.tune_variants(batch.scoring)


def _read(path, batch):
    with A.Context(0, autotune=True, tune_cache_path=str(path)) as ctx:
        return ctx.tune_variants(batch.scoring)


def test_a_file_of_another_build_is_not_read(tmp_path):
    path = tmp_path / "tune.txt"
    batch = W.make_config("small", n_pairs=64)
    chosen = _tuned(path, batch)
    lines = path.read_text().splitlines()
    assert lines[-1].startswith("build ") and _read(path, batch) == chosen
    key = lines[0].split()[0]
    path.write_text(f"{key} 1 1 1 1 0\n{lines[-1]}\n")                 # this build's
    assert _read(path, batch) == [1, 1, 1, 1, 0]
    path.write_text(f"{key} 1 1 1 1 0\nbuild another\n")               # another's
    assert _read(path, batch) is None
    assert _tuned(path, batch) is not None                             # measured again, written over
    assert path.read_text().splitlines()[-1] == lines[-1]
    path.write_text(f"{key} 1 1 1 1 0\n")                              # written by hand
    assert _read(path, batch) == [1, 1, 1, 1, 0]
