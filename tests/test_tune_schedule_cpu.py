"""What the schedule autotuner offers and remembers, with a fake timer (no GPU)."""
import os
import shutil

from paper_2010_03598_gb300 import api as A
from paper_2010_03598_gb300 import tune


def batch(path, timer):
    chains = [A.ChainSpec(L, 1.0, 0.5) for L in (10, 12, 14)]
    return tune.tune_batch(chains, A.Options(8, 0.05, 8), None, None, None, cache_path=path, timer=timer, gpu="g", sms=152)


def test_the_librarys_own_batch_schedule_is_timed_and_can_win(tmp_path):
    # ctas = tiles_per_cta = 0 is the one schedule that runs one launch per chain length
    seen = []

    def timer(cand):
        seen.append(dict(cand))
        return 55.0 if cand == dict(ctas=0, tiles_per_cta=0) else 114.0

    best = batch(str(tmp_path / "c.json"), timer)
    assert dict(ctas=0, tiles_per_cta=0) in seen
    assert (best["ctas"], best["tiles_per_cta"]) == (0, 0)
    assert len(seen) == 1 + len(tune.batch_candidates(152))


def test_a_schedule_of_another_build_is_timed_again(tmp_path, monkeypatch):
    # A cached choice was made between the kernels of its time: another version of the library's sources
    # may run other kernels for the same schedule.
    path, calls = str(tmp_path / "c.json"), []

    def timer(cand):
        calls.append(cand)
        return 1.0

    batch(path, timer)
    n = len(calls)
    batch(path, timer)
    assert len(calls) == n
    sources = tmp_path / "csrc"
    shutil.copytree(os.path.join(os.path.dirname(tune.__file__), "csrc"), sources)
    (sources / "kg_tile.cu").write_text((sources / "kg_tile.cu").read_text() + "// changed\n")
    monkeypatch.setattr(tune, "SOURCES", str(sources))
    tune.library_version.cache_clear()
    try:
        batch(path, timer)
    finally:
        tune.library_version.cache_clear()
    assert len(calls) == 2 * n
