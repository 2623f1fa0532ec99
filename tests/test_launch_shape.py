"""The autotuner knows which batches have a launch shape: its rule and limits are those of the library's sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_13245_gb300", "csrc")


def test_limits_are_the_librarys():
    from paper_2502_13245_gb300 import autotune
    src = open(os.path.join(CSRC, "rr_internal.h")).read()
    assert autotune.BEAM_CTA_QUERIES == int(re.search(r"kBeamCta2 = (\d+)", src).group(1))
    assert autotune.BEAM_CTA_BEAM == int(re.search(r"kBeamCtaBeam = (\d+)", src).group(1))


def test_small_batches_are_not_tuned():
    from paper_2502_13245_gb300.autotune import shape_matters, tune
    assert not shape_matters(1216, 32, "greedy") and not shape_matters(1, 512, "beam_es", {"es_metric": 1})
    assert shape_matters(1217, 32, "greedy") and shape_matters(1216, 31, "greedy")
    for p in ({"precision": 1}, {"expand": 2}, {"collect_stats": 1}, {"es_metric": 2}):
        assert shape_matters(100, 64, "greedy_es", p)
    assert not shape_matters(100, 64, "greedy", {"es_metric": 2})  # no early stop: the metric is not looked at

    class Q:
        shape = (100, 8)

    assert tune(None, Q, 1.0, "greedy", 64) == ({"tile_hint": 0, "seen_log2": 0, "persistent": 0}, [])
