"""The benchmark prints one JSON line that a log's tail still holds: the
autotuner's part of it names what was picked and each tile shape's total, not the
time of every variant, and no number has more than seven digits."""
import json

import bench


def test_the_autotuners_part_is_short():
    ms = {str(v): 3.141592653589793 for v in range(24)}
    tuned = dict(tile=[32, 16], fwd=7, bwd=9,
                 candidates={f"{w}x{h}": dict(total_ms=2.718281828, binning_ms=0.5, fwd=7, bwd=9, fwd_ms=ms, bwd_ms=ms)
                             for w, h in ((8, 8), (16, 8), (16, 16), (32, 16), (32, 32), (64, 32))})
    line = bench.tuned_summary(tuned)
    assert (line["tile"], line["fwd"], line["bwd"]) == ([32, 16], 7, 9)
    assert line["candidates"] == {t: 2.718281828 for t in tuned["candidates"]}
    assert len(json.dumps(bench.printed(line))) < 200 < len(json.dumps(tuned))
    assert tuned["candidates"]["8x8"]["fwd_ms"] is ms  # the caller's own is left whole
    assert bench.tuned_summary(None) is None
    given = {"tile": [16, 16], "fwd": 7, "bwd": 9, "given": True}
    assert bench.tuned_summary(given) == given


def test_numbers_of_seven_digits():
    x = {"a": 1944.4718775409842, "b": [1e-9 / 3, 13188101, True, None, "s"], "c": (2.0,)}
    assert bench.printed(x) == {"a": 1944.472, "b": [3.333333e-10, 13188101, True, None, "s"], "c": [2.0]}
    assert bench.printed(x)["b"][2] is True
