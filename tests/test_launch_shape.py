"""The autotuner knows which batches have a launch shape: its rule and limits are those of the library's sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_13245_gb300", "csrc")


def test_limits_are_the_librarys():
    from paper_2502_13245_gb300 import autotune
    src = open(os.path.join(CSRC, "rr_internal.h")).read()

    def value(name):
        return int(re.search(name + r" = (\d+)", src).group(1))

    assert autotune.BEAM_CTA_QUERIES == (value("kBeamCta4"), value("kBeamCta2"))
    assert autotune.BEAM_CTA_BEAM == value("kBeamCtaBeam")
    assert autotune.BEAM_CTA_LONG == (value("kBeamCta2Int"), value("kBeamCta2F32"))


def test_small_batches_are_not_tuned():
    from paper_2502_13245_gb300.autotune import shape_matters, tune
    assert not shape_matters(1216, 32, "greedy") and not shape_matters(1, 512, "beam_es", {"es_metric": 1})
    assert shape_matters(1217, 32, "greedy") and shape_matters(1216, 31, "greedy")
    assert not shape_matters(1216, 128, "greedy") and shape_matters(609, 129, "greedy")
    assert not shape_matters(608, 129, "greedy") and not shape_matters(1216, 256, "greedy", fp32=True)
    assert shape_matters(609, 257, "greedy", fp32=True)
    for p in ({"precision": 1}, {"expand": 2}, {"collect_stats": 1}, {"es_metric": 2}):
        assert shape_matters(100, 64, "greedy_es", p)
    assert not shape_matters(100, 64, "greedy", {"es_metric": 2})  # no early stop: the metric is not looked at

    class Q:
        shape = (100, 8)

    class Index:
        class info:
            dtype = 0

    assert tune(Index, Q, 1.0, "greedy", 64) == ({"tile_hint": 0, "seen_log2": 0, "persistent": 0}, [])
