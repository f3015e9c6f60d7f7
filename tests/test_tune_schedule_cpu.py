"""What the schedule autotuner offers and remembers, with a fake timer (no GPU)."""
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
